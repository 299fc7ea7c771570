"""The one-launch operator's first pass: which column and parity a group of threads
takes.  Every column once per parity, and one parity to a warp (the line transform
branches on it), for every number of columns a block can have.  Host program; no GPU."""
import os
import subprocess

import pytest

import test_fac_layout as layout

PROGRAM = r"""
#include "fft.cuh"
using namespace lsw;
template <int LOGN> int check() {
    constexpr int T = LineCfg<LOGN>::T, LINES = 256 / T, WARP = 32 / T;
    for (int cols = 1; cols <= 128; cols *= 2) {
        int seen[2][128] = {};
        for (int l0 = 0; l0 < parity_lines(cols, T); l0 += LINES)
            for (int g = 0; g < LINES; ++g) {
                int par, col, first, ignored;
                const bool valid = parity_line(l0 + g, cols, T, par, col);
                parity_line(l0 + g / WARP * WARP, cols, T, first, ignored);
                if (par != first) return 1;
                if (valid && (col < 0 || col >= cols || ++seen[par][col] != 1)) return 2;
            }
        for (int p = 0; p < 2; ++p)
            for (int c = 0; c < cols; ++c)
                if (seen[p][c] != 1) return 3;
    }
    return 0;
}
int main() { return check<3>() + 10 * check<4>() + 20 * check<5>() + 40 * check<6>() + 80 * check<7>(); }
"""


def test_one_parity_per_warp(tmp_path):
    nvcc = layout._nvcc()
    if not nvcc:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "lines.cu", tmp_path / "lines"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-arch=sm_103a", "-I", os.path.join(layout.ROOT, "include"),
                        "-I", os.path.join(layout.ROOT, "paper_2005_01372_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    assert subprocess.run([str(exe)]).returncode == 0
