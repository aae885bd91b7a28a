"""The tile shape that a plan of an FP64 batch asks for is the one that its per-step form runs: only the
initial shape, 32x8, is cut into smaller tiles, by the rule of lbm_launch.cuh (host code, compiled here)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r'''
#include <cstdio>
#include "lbm_launch.cuh"
int main()
{
    using namespace lbm;
    const int kinds[3] = {TILE_32x8, TILE_64x4, TILE_16x16};
    const long long sizes[4][2] = {{1, 8}, {69, 500}, {200, 1500}, {40000, 320000}};   // tiles, tiles of 8x4
    for (int k : kinds)
        for (auto& s : sizes)
            std::printf("%d ", fp64_batch_subtiles(k, s[0], s[1], 152) ? 1 : 0);
    for (auto& s : sizes) std::printf("%d ", fp64_small_tiles(s[0], s[1], 152) ? 1 : 0);
}
'''


def test_only_the_initial_shape_is_cut(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "paper_2603_22902_gb300", "csrc"), "-o", str(exe), str(src)],
                   check=True, capture_output=True)
    out = [int(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    rule = out[12:]
    assert out[:4] == rule and 0 < sum(rule) < 4      # 32x8: the rule of a single lattice, which takes either side here
    assert out[4:12] == [0] * 8                       # 64x4 and 16x16 as asked for
