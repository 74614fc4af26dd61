"""The rules that choose between the forms of the photon pools, compiled for the
CPU: they go by what the times go by (a cell's edge in mm), not by a cell's voxels."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1204_6367_gb300", "csrc")


def _evaluate(tmp_path, expressions):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    lines = "\n".join(f'    std::printf("%g\\n", (double)({e}));' for e in expressions)
    src.write_text('#include <cstdio>\n#include "transport_rules.h"\nusing namespace gdrr;\n'
                   "static float edge(float x, float y, float z, int s) { const float v[3] = {x, y, z}; "
                   "return cell_edge(v, s); }\nint main() {\n" + lines + "\n}\n")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True)
    return [float(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]


# voxel edge, cell shift, cell edge: the default cells are 32 mm whatever the voxel
CELLS = [(0.5, 6, 32.0), (1.0, 5, 32.0), (2.0, 4, 32.0), (4.0, 3, 32.0), (8.0, 2, 32.0), (1.0, 6, 64.0), (2.0, 5, 64.0),
         (4.0, 4, 64.0), (8.0, 3, 64.0), (16.0, 2, 64.0), (2.0, 6, 128.0), (8.0, 4, 128.0)]


def test_local_majorants_in_place_by_the_cells_edge(tmp_path):
    got = _evaluate(tmp_path, [f"lm_in_place(edge({v}f, {v}f, {v}f, {s}))" for v, s, _ in CELLS])
    assert got == [float(mm >= 64.0) for _, _, mm in CELLS]
    # the smallest edge counts
    assert _evaluate(tmp_path, ["edge(2.0f, 3.0f, 1.0f, 5)", "edge(4.0f, 2.0f, 8.0f, 3)"]) == [32.0, 16.0]


def test_coarse_cells_in_place_by_their_edge(tmp_path):
    cells = CELLS + [(3.0, 5, 96.0), (5.0, 5, 160.0), (3.0, 6, 192.0), (16.0, 4, 256.0), (4.0, 1, 8.0)]
    got = _evaluate(tmp_path, [f"coarse_in_place(edge({v}f, {v}f, {v}f, {s}))" for v, s, _ in cells])
    assert got == [float(mm >= 128.0) for _, _, mm in cells]


@pytest.mark.parametrize("nm", [2, 4, 8])
@pytest.mark.parametrize("gen", [0, 1])
@pytest.mark.parametrize("lm", [0, 1])
def test_default_pools_leave_the_sm_its_l1(tmp_path, nm, gen, lm):
    n, held, aligned = _evaluate(tmp_path, [f"default_pool({nm}, {gen}, {lm})",
                                            f"shared_of_blocks(default_pool({nm}, {gen}, {lm}), {nm}, {gen}, {lm})",
                                            f"pool_bytes(default_pool({nm}, {gen}, {lm}), {nm}, {gen}, {lm}) % 16"])
    # 256 KB of L1 and shared memory per SM, 60 KB of it L1; a pool is more than a
    # warp, its slots count in bytes, and the next warp's slots stay aligned
    assert held <= 196 * 1024 and 32 < n <= 84 and aligned == 0
    if (nm, gen, lm) == (4, 0, 0):
        assert n == 80
