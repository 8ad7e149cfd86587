"""The end of a persistent run, decided from the queue's counters (CPU).

A run has ended when every reserved slot is done.  Each electron adds its
children to `tail` before it adds itself to `done`, so tail >= done holds at
every moment and equality means the end; but a worker reads the two words at
different moments.  Every pair of moments is tried on short histories of the
counters: two reads in no particular order are fooled, the decision of
gt_queue.h is not.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "gt_queue.h"

// usage: harness <tail adds before each done add...>; prints the number of
// false ends and of true ends, for the plain comparison and for run_ended
int main(int argc, char **argv)
{
    unsigned long long tail[256], done[256];
    int n = 0;
    tail[0] = 1; done[0] = 0; ++n;  // one primary
    for (int i = 1; i < argc; ++i) {
        for (int k = atoi(argv[i]); k > 0; --k, ++n) { tail[n] = tail[n - 1] + 1; done[n] = done[n - 1]; }
        tail[n] = tail[n - 1]; done[n] = done[n - 1] + 1; ++n;
    }
    const bool over = tail[n - 1] == done[n - 1];
    int plain = 0, wrong = 0, right = 0;
    for (int a = 0; a < n; ++a)            // tail as polled
        for (int b = 0; b < n; ++b) {      // done as polled
            plain += tail[a] == done[b] && !(over && (b == n - 1));
            for (int c = (a > b ? a : b); c < n; ++c)   // the ordered pair, later
                for (int d = c; d < n; ++d) {
                    const bool end = gt::run_ended(tail[a], done[b], [&] { return done[c]; },
                                                   [&] { return tail[d]; });
                    if (end && !(over && c == n - 1)) ++wrong;
                    if (end && over && c == n - 1) ++right;
                }
        }
    printf("%d %d %d\n", plain, wrong, right);
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("queue_end")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I",
                    os.path.join(ROOT, "paper_2509_15377_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    return str(exe)


# children of each electron, in the order in which the electrons finish; the
# last history has not ended (one electron still flies)
@pytest.mark.parametrize("children,over", [((0,), True), ((1, 0), True), ((2, 0, 0), True),
                                           ((1, 1, 1, 0), True), ((3, 0, 2, 0, 0, 0), True),
                                           ((1, 1), False)])
def test_no_false_end(harness, children, over):
    out = subprocess.run([harness, *map(str, children)], check=True, capture_output=True,
                         text=True).stdout
    plain, wrong, right = map(int, out.split())
    assert wrong == 0
    assert (right > 0) == over  # a run that is over ends
    if max(children) > 0:
        assert plain > 0        # what the ordered pair is for
