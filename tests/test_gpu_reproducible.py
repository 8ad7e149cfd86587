"""Mixed precision, bit for bit: a run gives the same electrons again and with
every launch shape, for both gases and every option that has builds of its own
(the warp's vote and the build choose the code path, never the rounding)."""
import numpy as np
import pytest

from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W
from tests.gpu_helpers import by_uid, run_gpu

pytestmark = pytest.mark.gpu

SIGNAL = dict(signal_kind=W.W_PLATE, signal_bins=500, signal_dt=0.05)


@pytest.mark.parametrize("gas", ["basic", "physical"])
@pytest.mark.parametrize("option", [{}, {"crossing": 1}, SIGNAL, {"crossing": 1, **SIGNAL}])
@pytest.mark.parametrize("majorant", [A.GT_MAJORANT_GLOBAL, A.GT_MAJORANT_BANDED])
def test_same_electrons_again_and_with_every_shape(gas, option, majorant):
    import __graft_entry__
    __graft_entry__.build()
    w = W.plate(n_avalanches=40, seed=9)
    if gas == "physical":
        w.gas = W.argon_like_physical_gas()
    av = A.Avalanche(0)
    av.set_gas(w.gas)
    av.set_field(w.field)
    runs = [by_uid(run_gpu(av, w, seed=9, precision=A.GT_MIXED, majorant=majorant,
                           capacity=400_000, block=b, **option)[1])
            for b in (0, 0, 512, 768, 896, 1024)]
    av.close()
    assert len(runs[0]["uid"]) > 1000
    for r in runs[1:]:
        for k in ("uid", "status", "n_flight", "x0", "e0", "x1", "y1", "z1", "t1", "e1", "tallies"):
            assert np.array_equal(r[k], runs[0][k]), k


@pytest.mark.parametrize("gas", ["drift", "argon"])
@pytest.mark.parametrize("phase", [2, 6])
def test_global_majorant_build_equals_the_general_one(gas, phase):
    """In the unbounded uniform field the option of exact crossings changes
    nothing but the build: the global majorant's own and the general one give
    the same electrons bit for bit."""
    import __graft_entry__
    __graft_entry__.build()
    w = W.drift_model(n_electrons=100, n_coll=500, e_field=20_000.0, seed=12)
    if gas == "argon":
        w.gas = W.argon_like_gas()
    av = A.Avalanche(0)
    av.set_gas(w.gas)
    av.set_field(w.field)
    a, b = (by_uid(run_gpu(av, w, seed=12, precision=A.GT_MIXED, majorant=A.GT_MAJORANT_GLOBAL,
                           flights_per_phase=phase, capacity=400_000, crossing=c)[1])
            for c in (0, 1))
    av.close()
    for k in ("uid", "status", "n_flight", "x0", "x1", "y1", "z1", "t1", "e1", "tallies"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("tilt", [(0.0, 0.0, 1.0), (0.0, 0.0, -2.5)])
def test_tube_build_with_b_equals_the_general_one(tilt):
    """The tube's own build for B needs band bounds that rise with energy; a gas
    whose last band (99-100 eV, beyond every electron here) falls takes the
    build for any run, with the same bounds below."""
    import __graft_entry__
    __graft_entry__.build()
    w = W.coax(n_avalanches=64, r_lo=0.01, r_hi=0.03, seed=13)
    w.field.b = tilt
    av = A.Avalanche(0)
    runs = []
    for falling in (False, True):
        g = W.argon_like_gas()
        if falling:
            g.rate[1980:, 0] = 0.0
        av.set_gas(g)
        av.set_field(w.field)
        runs.append(by_uid(run_gpu(av, w, seed=13, precision=A.GT_MIXED, majorant=1,
                                   t_max=0.5, capacity=400_000)[1]))
    av.close()
    assert len(runs[0]["uid"]) >= 64 and max(r["e1"].max() for r in runs) < 95.0
    for k in ("uid", "status", "n_flight", "x0", "x1", "y1", "z1", "t1", "e1", "tallies"):
        assert np.array_equal(runs[0][k], runs[1][k]), k
