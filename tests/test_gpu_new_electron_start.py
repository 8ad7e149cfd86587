"""New electrons start inside the volume: their parent's boundary test decided
the same point, so the kernels test the start of primaries only.  Every kind
of boundary, both precisions, both structures of a run, a mesh with a hole."""
import math

import numpy as np
import pytest

import oracle
from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W
from tests.gpu_helpers import run_gpu

pytestmark = pytest.mark.gpu


def _workload(kind):
    if kind == "plate":
        return W.plate(n_avalanches=24, e_field=45_000.0, seed=31)
    w = W.coax(n_avalanches=24, b_axial=0.0, seed=31)
    phi = np.random.default_rng(31).uniform(0.0, 2.0 * math.pi, 24)
    w.primaries.x[:], w.primaries.y[:] = 0.008 * np.cos(phi), 0.008 * np.sin(phi)
    w.primaries.z[:] = 0.025
    if kind == "grid":
        w.field = W.coax_grid_map(n=65, half_width=0.02, length=0.05)
    elif kind == "mesh":
        f = W.coax_mesh_map(cells=6, half_width=0.02, length=0.05, seed=31)
        c = f.mesh_nodes[f.mesh_tets].mean(axis=1)
        hole = (c[:, 0] > 0.0) & (c[:, 1] > 0.0) & (np.hypot(c[:, 0], c[:, 1]) < 0.0075)
        f.mesh_tets = np.ascontiguousarray(f.mesh_tets[~hole])
        w.field = f
    return w


@pytest.mark.parametrize("mode", [A.GT_BATCHED, A.GT_PLAIN])
@pytest.mark.parametrize("precision", [A.GT_FP64, A.GT_MIXED])
@pytest.mark.parametrize("kind", ["plate", "coax", "grid", "mesh"])
def test_new_electrons_start_inside(kind, precision, mode):
    import __graft_entry__
    __graft_entry__.build()
    w = _workload(kind)
    n = w.primaries.n
    w.primaries.z[0] = -0.01 if kind == "plate" else w.primaries.z[0]
    if kind in ("grid", "mesh"):
        w.primaries.x[0] = 0.03   # a primary outside the volume ends where it starts
    elif kind == "coax":
        w.primaries.x[0], w.primaries.y[0] = 0.6, 0.0
    av = A.Avalanche(0)
    av.set_gas(w.gas)
    av.set_field(w.field)
    st, out = run_gpu(av, w, seed=31, precision=precision, mode=mode, majorant=1, t_max=1.0,
                      capacity=400_000)
    av.close()
    assert out["n_flight"][0] == 0 and out["status"][0] not in (0, W.TIME)
    assert np.all(out["n_flight"][n:] > 0) and st["n_endpoints"] > 2 * n
    r0 = np.stack([out["x0"], out["y0"], out["z0"]], axis=1)[n:]
    pick = np.random.default_rng(1).choice(len(r0), min(len(r0), 300), replace=False)
    assert all(oracle.boundary(w.field, r) == 0 for r in r0[pick])
