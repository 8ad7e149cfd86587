"""Division by a divisor known in advance (gt_math.h): the bits of an IEEE
division, over the operands of the magnetic step and at their edges (CPU)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "gt_math.h"

static uint64_t state = 1;
static uint32_t rnd()   // SplitMix64 (Steele, Lea, Flood, 2014)
{
    uint64_t z = state += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return (uint32_t)((z ^ (z >> 31)) >> 32);
}
static float make(int e, uint32_t m, uint32_t sign)
{
    uint32_t u = sign << 31 | (uint32_t)(e + 127) << 23 | (m & 0x7FFFFFu);
    float f;
    memcpy(&f, &u, 4);
    return f;
}

// usage: harness <lowest> <highest exponent> <divisor mantissa, or -1: any> <count>
int main(int, char **a)
{
    const int lo = atoi(a[1]), n = atoi(a[2]) - lo + 1;
    const long mant = atol(a[3]), count = atol(a[4]);
    long bad = 0;
    for (long i = 0; i < count; ++i) {
        const uint32_t w = rnd();
        const float d = make(lo + (int)(rnd() % n), mant < 0 ? rnd() : (uint32_t)mant, 0);
        const float x = make(lo + (int)(rnd() % n), rnd(), w & 1u);
        const volatile float want = x / d, r = 1.0f / d;
        bad += gt::div_known32(x, d, r) != want;
    }
    printf("%ld\n", bad);
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("known_divisor")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2509_15377_gb300", "csrc"), str(src), "-o",
                    str(exe), "-lm"], check=True)
    return str(exe)


# any divisor, a power of two, its neighbours, all ones
@pytest.mark.parametrize("mantissa", [-1, 0, 1, 0x7FFFFE, 0x7FFFFF, 0x400000, 0x555555])
@pytest.mark.parametrize("lo,hi", [(-3, 3), (-27, 27), (-48, 48)])
def test_bits_of_a_division(harness, lo, hi, mantissa):
    out = subprocess.run([harness, str(lo), str(hi), str(mantissa), "1000000"], check=True,
                         capture_output=True, text=True).stdout
    assert int(out) == 0
