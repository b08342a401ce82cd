"""Rows of the kernels that give each one several threads: the index in 64 bits up to
2^29 rows (the most a caller's matrix can have), and no kernel of the setup that
forms it in 32, where 32 threads to a row wrap at 2^27."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2311_13914_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <initializer_list>
#include "grid_index.h"
template <int SHIFT> long check(long long rows)
{
    const unsigned dim = 256;
    const long long per = dim >> SHIFT, blocks = (rows + per - 1) / per;
    long bad = 0;
    const long long at[] = {0, 1, rows / 2, (1LL << 27) - 1, 1LL << 27, (1LL << 27) + 5, rows - 1};
    for (long long r : at) {
        if (r >= rows) continue;
        const long long first = r << SHIFT;
        for (int k = 0; k < 1 << SHIFT; k++) {
            const long long block = (first + k) / dim;
            bad += block >= blocks || bd::grid_row<SHIFT>((unsigned)block, dim, (unsigned)((first + k) % dim)) != r;
        }
    }
    return bad;
}
int main()
{
    long bad = 0;
    for (long long rows : {1LL, 255LL, (1LL << 27) - 1, 1LL << 27, (1LL << 27) + 6, 1LL << 29})
        bad += check<5>(rows) + check<3>(rows);
    printf("%ld\n", bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_rows_beyond_32_bit_indices(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


@pytest.mark.parametrize("unit", ["amg_setup.cu", "bd_assemble.cu"])
def test_no_setup_kernel_divides_a_32_bit_index(unit):
    text = open(os.path.join(CSRC, unit)).read()
    assert not re.findall(r"\(blockIdx\.x \* blockDim\.x \+ threadIdx\.x\)\s*(?:>>|/)[^\n]*", text)
