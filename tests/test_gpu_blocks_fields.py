"""Mixed precision, bit for bit: at a fixed refill period a run gives the same
electrons with every number of threads per CTA, in every kind of field, with
magnetic fields along an axis and tilted, for both gases and majorants (the
plate without B: test_gpu_reproducible.py)."""
import numpy as np
import pytest

from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W
from tests.gpu_helpers import by_uid, run_gpu

pytestmark = pytest.mark.gpu


def _workload(kind, n=24):
    if kind == "plate":
        return W.plate(n_avalanches=n, seed=17)
    if kind == "uniform":
        w = W.drift_model(n_electrons=n, n_coll=300, e_field=20_000.0, seed=17)
        w.gas = W.argon_like_gas()
        return w
    w = W.coax(n_avalanches=n, b_axial=0.0, seed=17)
    phi = np.random.default_rng(17).uniform(0.0, 2.0 * np.pi, n)
    w.primaries.x[:], w.primaries.y[:] = 0.009 * np.cos(phi), 0.009 * np.sin(phi)
    w.primaries.z[:] = 0.025
    if kind == "grid":
        w.field = W.coax_grid_map(n=65, half_width=0.02, length=0.05)
    elif kind == "mesh":
        w.field = W.coax_mesh_map(cells=6, half_width=0.02, length=0.05, seed=17)
    return w


@pytest.mark.parametrize("majorant", [A.GT_MAJORANT_GLOBAL, A.GT_MAJORANT_BANDED])
@pytest.mark.parametrize("gas", ["basic", "physical"])
@pytest.mark.parametrize("b", [(0.0, 0.0, 0.0), (0.0, 0.0, 1.0), (0.7, -0.4, 1.1)])
@pytest.mark.parametrize("kind", ["plate", "uniform", "coax", "grid", "mesh"])
def test_same_electrons_with_every_block(kind, b, gas, majorant):
    import __graft_entry__
    __graft_entry__.build()
    w = _workload(kind)
    if gas == "physical":
        w.gas = W.argon_like_physical_gas()
    w.field.b = b
    av = A.Avalanche(0)
    av.set_gas(w.gas)
    av.set_field(w.field)
    runs = [by_uid(run_gpu(av, w, seed=17, t_max=0.3, precision=A.GT_MIXED, majorant=majorant,
                           capacity=400_000, refill_period=16, block=t)[1])
            for t in (512, 768, 896, 1024)]
    av.close()
    assert len(runs[0]["uid"]) >= 24
    for r in runs[1:]:
        for k in ("uid", "status", "n_flight", "x0", "e0", "x1", "y1", "z1", "t1", "e1", "tallies"):
            assert np.array_equal(r[k], runs[0][k]), k


@pytest.mark.parametrize("b", [(0.7, -0.4, 1.1), (0.0, 0.9, 0.0), (-1.3, 0.2, 0.1)])
def test_tube_build_with_tilted_b_equals_the_general_one(b):
    """The tube's own build for B needs band bounds that rise with energy; a gas
    whose last band (99-100 eV, beyond every electron here) falls takes the
    build for any run, with the same bounds below."""
    import __graft_entry__
    __graft_entry__.build()
    w = _workload("coax", n=64)
    w.field.b = b
    av = A.Avalanche(0)
    runs = []
    for falling in (False, True):
        g = W.argon_like_gas()
        if falling:
            g.rate[1980:, 0] = 0.0
        av.set_gas(g)
        av.set_field(w.field)
        runs.append(by_uid(run_gpu(av, w, seed=17, precision=A.GT_MIXED, majorant=1, t_max=0.5,
                                   capacity=400_000)[1]))
    av.close()
    assert max(r["e1"].max() for r in runs) < 95.0
    for k in ("uid", "status", "n_flight", "x0", "x1", "y1", "z1", "t1", "e1", "tallies"):
        assert np.array_equal(runs[0][k], runs[1][k]), k
