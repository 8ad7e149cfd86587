"""FP64 runs at the edges of the level search and of the plain mode's split of a
generation over SMs, warps and lanes, electron by electron."""
import numpy as np
import pytest

import oracle
from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W
from tests.gpu_helpers import assert_same_electrons, by_uid, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def av():
    import __graft_entry__
    __graft_entry__.build()
    a = A.Avalanche(0)
    yield a
    a.close()


def _gas(levels):
    """Elastic level first, then excitations, one ionisation last; rates that
    vary with energy and vanish below threshold, so that running sums repeat."""
    n, d_eps = 401, 0.1
    eps = np.arange(n) * d_eps
    types, thr, cols = [W.ELASTIC], [0.0], [300.0 * np.sqrt(eps)]
    for j in range(1, levels):
        e = 4.0 + 8.0 * j / levels
        types.append(W.IONISATION if j == levels - 1 else W.EXCITATION)
        thr.append(e)
        cols.append(np.where(eps >= e, (40.0 + 7.0 * (j % 5)) * (eps - e), 0.0))
    return W.Gas(np.array(types, np.int32), np.array(thr), np.stack(cols, axis=1), d_eps, 2e-5)


@pytest.mark.parametrize("levels", [1, 2, 3, 4, 9, 16, 17, 31, 32])
@pytest.mark.parametrize("majorant", [A.GT_MAJORANT_GLOBAL, A.GT_MAJORANT_BANDED])
def test_levels(av, levels, majorant):
    w = W.plate(n_avalanches=30, e_field=30_000.0, seed=levels)
    w.gas = _gas(levels)
    av.set_gas(w.gas)
    av.set_field(w.field)
    _, out = run_gpu(av, w, seed=3, t_max=0.1, majorant=majorant, capacity=1_000_000)
    ref = oracle.run(w.gas, w.field, w.primaries, seed=3, t_max=0.1, majorant=majorant)
    assert_same_electrons(out, ref, scale_pos=0.0128, scale_t=0.1)
    assert np.array_equal(out["tallies"], ref["tallies"])


@pytest.mark.parametrize("precision", [A.GT_FP64, A.GT_MIXED])
@pytest.mark.parametrize("n", [1, 2, 151, 153, 305, 609, 5000, 20_000])
def test_plain_generation_sizes(av, n, precision):
    """One avalanche of n primaries: n electrons in its first generation."""
    w = W.plate(n_avalanches=n, seed=n)
    w.primaries.aval[:] = 0
    w.primaries.n_avalanches = 1
    av.set_gas(w.gas)
    av.set_field(w.field)
    kw = dict(seed=4, t_max=0.02, majorant=1, precision=precision, capacity=4 * n + 64)
    if precision == A.GT_MIXED:
        kw["refill_period"] = 1 << 20  # the plain step never folds its offsets
    plain = by_uid(run_gpu(av, w, mode=A.GT_PLAIN, **kw)[1])
    batched = by_uid(run_gpu(av, w, mode=A.GT_BATCHED, **kw)[1])
    for k in ("uid", "status", "n_flight", "x0", "z0", "x1", "y1", "z1", "t1", "e1", "tallies"):
        if precision == A.GT_FP64 or k in ("uid", "status", "n_flight", "tallies"):
            assert np.array_equal(plain[k], batched[k]), k
