"""The default launch shape follows the size that a run may be expected to have
and the shared memory that its gas table leaves, not the capacity alone."""
import numpy as np
import pytest
import torch

from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIGNAL = dict(signal_kind=W.W_PLATE, signal_bins=100, signal_dt=0.05)


def _block(w, capacity, **kw):
    import __graft_entry__
    __graft_entry__.build()
    av = A.Avalanche(0)
    av.set_gas(w.gas)
    av.set_field(w.field)
    kw = dict(dict(precision=A.GT_MIXED, majorant=A.GT_MAJORANT_BANDED), **kw)
    # a short time limit: the shape is chosen before the run
    st = av.run(av.primaries_device(w.primaries), A.RunOptions(seed=1, t_max=0.01, **kw), capacity)
    av.close()
    return st["block"]


def _lanes():
    return 1024 * torch.cuda.get_device_properties(0).multi_processor_count


# (avalanches, V/cm, gap, room per lane, options, threads): few electrons in much room
# stay at 512 (the gains are about 10, 97, 320 and 996 at 20, 30, 35 and 40 kV/cm)
@pytest.mark.parametrize("n,e,gap,room,kw,want", [
    (400, 30e3, 0.0128, 40, {}, 512), (1000, 30e3, 0.0128, 40, {}, 512),
    (2301, 30e3, 0.0128, 10, {}, 512), (10000, 20e3, 0.0128, 40, {}, 512),
    (800, 35e3, 0.0128, 40, {}, 512), (1000, 3e3, 0.1, 40, {}, 512),
    (1000, 30e3, 0.0128, 40, {"crossing": 1}, 512), (1000, 30e3, 0.0128, 40, SIGNAL, 512),
    (1000, 40e3, 0.0128, 40, {"size_limit": 100}, 512),
    (1000, 40e3, 0.0128, 7.9, {}, 512), (1000, 40e3, 0.0128, 8, {}, 896),
    (1000, 40e3, 0.0128, 32, {}, 1024), (10000, 30e3, 0.0128, 8, {}, 896),
    (40000, 25e3, 0.0128, 32, {}, 1024), (1000, 40e3, 0.0128, 8, {"crossing": 1}, 768),
    (1000, 40e3, 0.0128, 32, {"crossing": 1}, 1024), (1000, 40e3, 0.0128, 32, SIGNAL, 768),
    (1000, 40e3, 0.0128, 32, {"majorant": A.GT_MAJORANT_GLOBAL}, 512),
    (1000, 40e3, 0.0128, 32, {"precision": A.GT_FP64}, 160)])
def test_follows_the_expected_size(n, e, gap, room, kw, want):
    assert _block(W.plate(n, e, gap=gap, seed=1), int(room * _lanes()), **kw) == want


def test_no_growth():
    """Without an ionisation that has a rate the primaries are the run."""
    silent = W.argon_like_gas()
    silent.rate[:, silent.level_type == W.IONISATION] = 0.0
    for gas in (W.model_gas(), silent):
        w = W.plate(1000, 40e3, seed=1)
        w.gas = gas
        assert _block(w, 32 * _lanes()) == 512


# levels, nodes -> the largest of 1024, 896, 768 and 512 threads whose state, counts and
# band table leave room for the gas table (1024 at 12 levels, 896 at 16, 768 at 17)
@pytest.mark.parametrize("levels,nodes", [(12, 2001), (13, 2001), (14, 2001), (15, 2001),
                                          (16, 2001), (17, 2001), (18, 1801), (20, 1601),
                                          (31, 1101), (32, 4001)])
def test_step_down_is_exact(levels, nodes):
    top = 100.0
    d_eps = top / (nodes - 1)
    eps = np.arange(nodes) * d_eps
    types = np.array([W.ELASTIC] + [W.EXCITATION] * (levels - 2) + [W.IONISATION], np.int32)
    thr = np.concatenate([[0.0], np.linspace(11.5, 15.0, levels - 2), [15.7]])
    cols = [1000.0 * np.sqrt(eps)] + [np.where(eps >= t, 5.0 * (eps - t), 0.0) for t in thr[1:]]
    w = W.plate(1000, 40e3, seed=1)
    w.gas = W.Gas(types, thr, np.stack(cols, axis=1), d_eps, 2e-5)
    per = max(1, int(np.floor(1.0 / d_eps + 0.5)))      # nodes per band of 1 eV
    bands = -(-(nodes - 1) // per)
    rows = bands.bit_length()                             # range maxima over 1, 2, 4, ... bands
    room = torch.cuda.get_device_properties(0).shared_memory_per_block_optin - 4096

    def align(b):
        return (b + 15) & ~15

    def fits(block):
        return (32 * block + align(4 * levels * block) + align(4 * bands * rows)
                + 4 * (levels | 1) * nodes) <= room

    want = next((b for b in (1024, 896, 768) if fits(b)), 512)
    assert _block(w, 32 * _lanes()) == want
