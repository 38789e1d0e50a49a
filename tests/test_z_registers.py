"""Registers of float z-line kernels, from the compiler's report: the R2C lines of 64 and
1024 reals keep four blocks of 256 threads an SM (64 registers), the looping C2R lines of
1536 reals two (128).  A __grid_constant__ argument costs them a block each (80 and 159)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2202_12756_gb300")

PROGRAM = r"""
#include "kern_impl.cuh"
using namespace fft3d;
void *const kernels[] = {(void *)z_kernel<float, 512, false, false, false>(), (void *)z_kernel<float, 32, false, false, false>(),
                         (void *)z_kernel<float, 768, true, true, false>()};
"""


def test_float_z_lines_keep_their_resident_blocks(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "z.cu"
    src.write_text(PROGRAM)
    out = subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a", "-Xptxas", "-v",
                          "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"), "-c", str(src),
                          "-o", str(tmp_path / "z.o")], check=True, capture_output=True, text=True, timeout=600).stderr
    regs = {}
    for name, n in re.findall(r"entry function '\S*(zpass_(?:r2c|c2r)_kernelIfLi\d+)\S*'.*?Used (\d+) registers", out, re.S):
        regs[name] = int(n)
    assert regs["zpass_r2c_kernelIfLi512"] <= 64
    assert regs["zpass_r2c_kernelIfLi32"] <= 64
    assert regs["zpass_c2r_kernelIfLi768"] <= 128
