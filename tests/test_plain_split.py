"""How a plain generation is split over SMs, warps and lanes (gt_plain.h, CPU):
every electron has one place, and a block launches all its threads, whose
surplus warps copy the gas table, however few electrons there are."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "gt_plain.h"

// usage: harness <electrons> <SMs> <threads>; the kernel's own index
int main(int, char **a)
{
    const long long n = atoll(a[1]);
    const int sms = atoi(a[2]), threads = atoi(a[3]);
    const gt::PlainSplit s = gt::plain_split(n, sms, threads);
    std::vector<int> seen((size_t)n, 0);
    for (unsigned b = 0; b < s.blocks; ++b)
        for (int t = 0; t < threads; ++t) {
            const int lane = t & 31, wid = t >> 5;
            const long long i = ((long long)b * s.warps + wid) * s.lanes + lane;
            if (wid >= s.warps || lane >= s.lanes || i >= n) continue;
            ++seen[(size_t)i];
        }
    int bad = 0;
    for (int c : seen) bad += c != 1;
    printf("%d %d %d %u\n", bad, s.warps, s.lanes, s.blocks);
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("plain_split")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I",
                    os.path.join(ROOT, "paper_2509_15377_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("threads", [32, 64, 128])
@pytest.mark.parametrize("n", [1, 2, 151, 152, 153, 304, 305, 608, 609, 4864, 4865, 9729, 19456,
                               19457, 100_003])
def test_every_electron_has_one_place(harness, n, threads):
    bad, warps, lanes, blocks = map(int, subprocess.run(
        [harness, str(n), "152", str(threads)], check=True, capture_output=True,
        text=True).stdout.split())
    assert bad == 0
    assert 1 <= warps <= threads // 32 and 1 <= lanes <= 32
    # SMs first, then warps, then lanes
    assert blocks >= min(n, 152) or warps > 1 or lanes > 1
    assert warps == min(-(-n // 152), threads // 32)
    assert lanes == 1 or n > 152 * warps * (lanes - 1)
