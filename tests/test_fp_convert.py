"""Integer float <-> double conversions against the compiler's, bit for bit: every
exponent, the mantissas around the rounding ties, and everything that is not normal."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2311_13914_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "fp_convert.h"
using namespace bd;
static uint64_t seed = 88172645463325252ull;
static uint64_t rnd() { seed ^= seed << 13; seed ^= seed >> 7; seed ^= seed << 17; return seed; }
int main()
{
    long bad = 0, n = 0;
    for (uint32_t se = 0; se < 512; se++)
        for (int k = 0; k < 64; k++) {
            const uint32_t man = k == 0 ? 0 : k == 1 ? 1 : k == 2 ? 0x7fffffu : k == 3 ? 0x400000u : (uint32_t)rnd() & 0x7fffffu;
            const uint32_t b = se << 23 | man;
            float f;
            memcpy(&f, &b, 4);
            bad += fp_bits(widen(f)) != fp_bits((double)f);
            n++;
        }
    const uint64_t half = 0x10000000ull;
    for (uint32_t se = 0; se < 4096; se++)
        for (int k = 0; k < 64; k++) {
            uint64_t man = rnd() & 0xfffffffffffffull;
            if (k < 32) {  // ties and their neighbours, below even and odd last bits
                const uint64_t top = k < 8 ? 0 : k < 16 ? 1 : k < 24 ? 0x7fffffull : man >> 29;
                const uint64_t low[8] = {0, 1, half - 1, half, half + 1, 2 * half - 1, rnd() & (2 * half - 1), half ^ 2};
                man = top << 29 | low[k & 7];
            }
            const uint64_t b = (uint64_t)se << 52 | man;
            double d;
            memcpy(&d, &b, 8);
            bad += fp_bits(narrow(d)) != fp_bits((float)d);
            n++;
        }
    printf("%ld of %ld\n", bad, n);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_conversions_equal_the_compilers(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
