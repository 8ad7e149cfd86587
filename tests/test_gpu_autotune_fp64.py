"""The FP64 tuner starts from the default shape: a tuned run has no slower one
than an untuned run by the tuner's own measurements, and uses what it chose."""
import pytest

from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("majorant", [A.GT_MAJORANT_GLOBAL, A.GT_MAJORANT_BANDED])
@pytest.mark.parametrize("fixed", [{}, {"block": 256}, {"refill_period": 16}])
def test_default_shape_is_measured(majorant, fixed):
    import __graft_entry__
    __graft_entry__.build()
    w = W.plate(n_avalanches=40, e_field=30_000.0, seed=21)
    av = A.Avalanche(0)
    av.set_gas(w.gas)
    av.set_field(w.field)
    p = av.primaries_device(w.primaries)
    opt = A.RunOptions(seed=21, t_max=0.2, precision=A.GT_FP64, majorant=majorant, **fixed)
    default = av.run(p, opt, 100_000)
    best, points = av.autotune(p, opt, capacity=100_000)
    tuned = av.run(p, opt, 100_000)
    av.close()
    shapes = {(q["block"], q["refill_period"]): q["real_per_ms"] for q in points}
    assert (default["block"], default["refill_period"]) in shapes
    assert best["real_per_ms"] >= shapes[default["block"], default["refill_period"]]
    assert (tuned["block"], tuned["refill_period"]) == (best["block"], best["refill_period"])
