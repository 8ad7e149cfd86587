"""The default launch shape of a mixed plate run with room for many electrons:
as many threads as the gas table leaves shared memory for, the same electrons
as with 512 threads, and no run refused that 512 threads take."""
import numpy as np
import pytest

from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W
from tests.gpu_helpers import by_uid, run_gpu

pytestmark = pytest.mark.gpu


def _gas(levels, nodes):
    eps = np.arange(nodes) * (100.0 / (nodes - 1))
    types = np.array([W.ELASTIC] + [W.EXCITATION] * (levels - 2) + [W.IONISATION], np.int32)
    thr = np.concatenate([[0.0], np.linspace(11.0, 15.0, levels - 2), [15.7]])
    cols = [1000.0 * np.sqrt(eps)] + [np.where(eps >= t, 5.0 * (eps - t), 0.0) for t in thr[1:]]
    return W.Gas(types, thr, np.stack(cols, axis=1), 100.0 / (nodes - 1), 2e-5)


@pytest.mark.parametrize("levels,nodes", [(12, 2001), (15, 2001), (17, 2001), (31, 1101),
                                          (32, 4001)])
@pytest.mark.parametrize("capacity", [1_000_000, 1_500_000, 6_000_000])
def test_default_shape(levels, nodes, capacity):
    import __graft_entry__
    __graft_entry__.build()
    w = W.plate(n_avalanches=400, seed=15)
    av = A.Avalanche(0)
    av.set_gas(_gas(levels, nodes))
    av.set_field(w.field)
    kw = dict(seed=15, t_max=0.1, precision=A.GT_MIXED, majorant=1, capacity=capacity)
    st, out = run_gpu(av, w, **kw)
    _, ref = run_gpu(av, w, block=512, **kw)
    av.close()
    # bytes per thread: FP64 bases 32, a count per level 4; the table's rows have odd length
    table = 4 * (levels | 1) * nodes
    fits = [b for b in (512, 768, 896, 1024) if b * (32 + 4 * levels) + table < 227_000]
    want = 512 if capacity < 1_245_184 else 896 if capacity < 4_980_736 else 1024
    assert st["block"] <= max([b for b in fits if b <= want], default=512)
    if levels == 12:
        assert st["block"] == want
    a, b = by_uid(out), by_uid(ref)
    for k in ("uid", "status", "n_flight", "x1", "z1", "e1", "tallies"):
        assert np.array_equal(a[k], b[k]), k
