"""Host rule of the tiles' depth (compiled here for the CPU): a block's planes come in
as many tiles as the depth asks for, all of them nearly equal."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "internal.cuh"
int main() {
    for (int nz = 1; nz <= 300; ++nz)
        for (int depth = 1; depth <= 32; depth *= 2)
            std::printf("%d %d %d\n", nz, depth, flosic::tile_split(nz, depth));
}
"""


def test_planes_are_split_evenly(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "split.cu", tmp_path / "split"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2108_01186_gb300", "csrc"), "-o", str(exe), str(src)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    for nz, depth, tz in zip(*(map(int, lines[k::3]) for k in range(3))):
        n = -(-nz // depth)
        assert 1 <= tz <= depth and -(-nz // tz) <= n
        assert tz == -(-nz // n)          # no tiles of n could have a smaller largest depth
