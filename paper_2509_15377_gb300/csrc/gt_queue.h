// gt_queue.h -- when a persistent run has ended.  Also compiled by the host
// compiler, which tries the decision on every pair of moments of its reads.
#pragma once

#include "gt_math.h"

namespace gt {

// Every reserved slot is done?  An electron's children are in `tail` before
// the electron is in `done` (push_children has its atomic's result back
// before the warp counts its finished electrons), so that tail never falls
// behind done and equal counts of one moment mean the end.  (tail, done) as
// polled are two words of no common moment: an older tail beside a newer done
// can be equal while a new electron waits.  They are a hint; the end is
// decided by a second pair, done read before tail, which in any interleaving
// can only see more slots than were reserved when done was read.  The second
// pair costs nothing while the run goes on.
template <class LoadDone, class LoadTail>
GT_HOST_DEVICE bool run_ended(unsigned long long tail, unsigned long long done,
                              LoadDone load_done, LoadTail load_tail)
{
    if (tail != done) return false;
    const unsigned long long d = load_done();
    return load_tail() == d;
}

}  // namespace gt
