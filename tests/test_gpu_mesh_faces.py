"""Mixed precision on a mesh: the electrons of a run whose elements are kept in
shared memory (512 threads) are those of a run that reads every record (1024
threads, where they do not fit)."""
import numpy as np
import pytest

from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W
from tests.gpu_helpers import by_uid, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grading", [0.0, 4.0])
@pytest.mark.parametrize("crossing", [0, 1])
def test_kept_elements_equal_records(grading, crossing):
    import __graft_entry__
    __graft_entry__.build()
    w = W.mesh_coax(n_avalanches=24, cells=2, seed=5)
    w.field = W.coax_mesh_map(cells=8, half_width=0.02, length=0.05, voltage=1500.0, seed=5,
                              grading=grading)
    w.gas = W.argon_like_physical_gas()
    ph = np.random.default_rng(5).uniform(0.0, 2.0 * np.pi, 24)
    w.primaries.x[:], w.primaries.y[:] = 0.012 * np.cos(ph), 0.012 * np.sin(ph)
    w.primaries.z[:] = 0.025
    av = A.Avalanche(0)
    av.set_gas(w.gas)
    av.set_field(w.field)
    runs = [by_uid(run_gpu(av, w, seed=5, precision=A.GT_MIXED, majorant=1, capacity=8_000_000,
                           crossing=crossing, block=b)[1]) for b in (512, 1024)]
    av.close()
    assert len(runs[0]["uid"]) > 200
    for k in ("uid", "status", "n_flight", "x0", "y1", "z1", "t1", "e1", "tallies"):
        assert np.array_equal(runs[0][k], runs[1][k]), k
