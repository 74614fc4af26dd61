"""Where the backprojection reads a group's samples untested, every row it reads
lies inside the detector.  The kernel's own expressions, compiled for the CPU with
contraction off, over columns whose first or last voxel falls within rounding of
row 0 or of the last row."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1204_6367_gb300", "csrc")

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include "fdk_rows.h"
using namespace gdrr;
static uint64_t state = 88172645463325252ull;
static double uniform() {
    state ^= state << 13; state ^= state >> 7; state ^= state << 17;
    return (state >> 11) * (1.0 / 9007199254740992.0);
}
int main() {
    long inside = 0, bad = 0;
    for (int i = 0; i < 4000000; ++i) {
        const int nv = 2 + (int)(uniform() * 400), iz0 = 4 * (int)(uniform() * 64);
        const float dz = (float)(0.1 + 4.0 * uniform()), sv = (float)(0.2 + 2.0 * uniform());
        const float hv = (float)(0.5 * nv - 0.5);
        // the first (last) voxel at row 0 (nv - 1), give or take a few roundings
        const bool low = uniform() < 0.5;
        const double z = ((low ? 0.0 : nv - 1.0) - hv) / sv;
        const float z0 = (float)(z - (iz0 + (low ? 0 : 3)) * (double)dz) * (float)(1.0 + (uniform() - 0.5) * 4e-7);
        const float lo = bp_row(bp_height(z0, iz0, dz), sv, hv), hi = bp_row(bp_height(z0, iz0 + 3, dz), sv, hv);
        if (!bp_rows_inside(lo, hi, nv)) continue;
        ++inside;
        for (int k = 0; k < 4; ++k) {
            // as the packed taps form it
            const float row = std::fmaf(std::fmaf((float)(iz0 + k), dz, z0), sv, hv);
            const int iv = (int)std::floor(row);
            if (iv < 0 || iv > nv - 2) { ++bad; break; }
        }
    }
    std::printf("%ld %ld\n", inside, bad);
    return 0;
}
"""


def test_rows_read_untested_are_inside(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    inside, bad = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert inside > 100_000
    assert bad == 0
