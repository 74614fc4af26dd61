"""The row filter's launch shape, compiled for the CPU: every row and task is
covered once, few rows spread over the SMs, many fill their blocks, and no shape
needs more shared memory than the limit that the kernel asks for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1204_6367_gb300", "csrc")
SMS = 152

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "fdk_filter.h"
int main(int argc, char** argv) {
    for (int i = 1; i + 2 < argc; i += 3) {
        const gdrr::FilterShape f = gdrr::filter_shape(std::atoi(argv[i]), std::atoll(argv[i + 1]), %d, std::atoi(argv[i + 2]) != 0);
        std::printf("%%d %%d %%d %%zu %%zu\n", f.rows, f.parts, gdrr::filter_tasks(f), gdrr::filter_smem(f), gdrr::filter_smem_most());
    }
}
""" % SMS


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("shape")
    (d / "shape.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "shape.cpp"), "-o", str(d / "shape")], check=True)

    def run(nu, n_rows, share=True):
        out = subprocess.run([str(d / "shape"), str(nu), str(n_rows), str(int(share))], check=True, capture_output=True, text=True)
        return [int(v) for v in out.stdout.split()]
    return run


@pytest.mark.parametrize("nu", [1, 8, 63, 64, 512, 1030, 4096])
@pytest.mark.parametrize("n_rows", [1, 8, 128, 768, 34_560, 138_240])
def test_rows_are_spread_and_blocks_filled(shape, nu, n_rows):
    rows, parts, tasks, smem, most = shape(nu, n_rows)
    blocks = -(-n_rows // rows)
    assert rows % 4 == 0 and 1 <= parts and smem <= most
    # no more rows a block than spread them over three blocks an SM
    assert rows == 4 or blocks * rows <= n_rows + rows and (rows - 4) * 3 * SMS < n_rows
    # a full call keeps blocks with a task for every thread
    if n_rows >= 138_240:
        assert tasks > 128 and parts == 1
    # shared rows only where SMs would stay idle
    assert parts == 1 or blocks * parts <= SMS
    assert shape(nu, n_rows, False)[1] == 1                # in place: a block owns its rows
