"""The output slice of a tcgen05 convolution (umma_slice in conv_umma.cuh): a fused input or head is
only ever given to the kernel that knows it, at 16 outputs a launch, and what a slice needs fits
shared memory.  Host code only, compiled and run without a GPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include <cstdio>
#include "conv_umma.cuh"
int main()
{
    for (int ci = 8; ci <= 192; ci += 8)
        for (int co = 8; co <= 128; co += 8)
            for (int f = 0; f < 2; ++f) {
                const int nt = pmeft::umma_slice(ci, co, f != 0);
                std::printf("%d %d %d %d %zu\\n", ci, co, f, nt, nt ? pmeft::umma_smem(nt, ci, 2) : (size_t)0);
            }
}
"""


def test_slices(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    (tmp_path / "s.cu").write_text(SRC)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", ROOT + "/include", "-I",
                    ROOT + "/paper_2604_15434_gb300/csrc", "-o", str(tmp_path / "s"), str(tmp_path / "s.cu")], check=True)
    out = subprocess.run([str(tmp_path / "s")], check=True, capture_output=True, text=True).stdout
    got = {tuple(map(int, line.split()[:3])): tuple(map(int, line.split()[3:])) for line in out.splitlines()}
    for (ci, co, fused), (nt, smem) in got.items():
        if ci % 16 or co % 16:
            assert nt == 0
        elif fused:
            assert nt in (0, 16)
        else:
            assert nt == 0 or (nt <= 64 and co % nt == 0)
        assert smem <= 227 * 1024
    # the network's layers: as given, and the four that a forward pass fuses
    layers = {(16, 16): 16, (16, 32): 32, (32, 32): 32, (32, 64): 64, (64, 64): 32, (96, 32): 16, (48, 16): 16,
              (32, 96): 48, (16, 48): 48}
    for (ci, co), nt in layers.items():
        assert got[ci, co, 0][0] == nt, (ci, co, got[ci, co, 0])
    for ci, co in ((16, 16), (96, 32), (48, 16)):
        assert got[ci, co, 1][0] == 16
