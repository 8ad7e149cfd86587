// gt_plain.h -- how a plain generation is split.  No CUDA: also compiled by
// the host compiler.
#pragma once

#include <algorithm>

namespace gt {

// Electron i sits in lane i % lanes of warp i / lanes, and a block's first
// `warps` warps hold electrons.
struct PlainSplit {
    int warps, lanes;
    unsigned blocks;
};

// A generation lasts as long as its longest chain of flights: its electrons
// spread over the SMs first, then over the warps of a block of `threads`, then
// over the warps' lanes.  (Blocks of 32 electrons per warp put a generation of
// 100 on one SM, whose FP64 pipe takes 16 clocks per warp instruction however
// many lanes are active: two FP64 avalanches of the 40 kV/cm plate 173 ms, now
// 112.)  A block keeps its other warps: they help to copy the mixed step's
// 96-KB gas table into shared memory, which every block does in every
// generation.  (Two mixed avalanches of the general gas in the tube, 318
// electrons: 6.5 ms with blocks of the electrons' warps alone, 4.0 with all of
// them; 4.4 with 32 electrons per warp.)
inline PlainSplit plain_split(long long n, int sms, int threads)
{
    PlainSplit s;
    s.warps = (int)std::min<long long>((n + sms - 1) / sms, threads / 32);
    const long long all = (long long)sms * s.warps;
    s.lanes = (int)std::min<long long>((n + all - 1) / all, 32);
    const long long per = (long long)s.lanes * s.warps;
    s.blocks = (unsigned)((n + per - 1) / per);
    return s;
}

}  // namespace gt
