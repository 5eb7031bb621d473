"""Registers of the FP64 stage kernels of the 16-point rules, from the compiler's
report: the grid of a right-hand side and of an RK stage alike counts on three blocks
on every SM, which 65536 registers hold up to 80 a thread with blocks of 8 warps and
168 with the right-hand side's blocks of 4."""

import os
import re
import shutil
import subprocess

import pytest

from paper_2005_02516_gb300 import _build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("unit", ["esdg_kernels_s4.cu", "esdg_kernels_n3.cu"])
def test_three_blocks_of_the_stage_kernels_fit(unit, tmp_path):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no CUDA compiler")
    p = subprocess.run([_build.nvcc(), "-c", os.path.join(_build.CSRC, unit), "-o", str(tmp_path / "o.o"), "-O3",
                        "-std=c++17", "-lineinfo", "-Xptxas", "-v", *_build.ARCH, "-I", _build.CSRC, "-I",
                        os.path.join(ROOT, "include")], capture_output=True, text=True, check=True)
    found = re.findall(r"entry function '_ZN4esdg7k_stageILi\d+EdLi(\d)E(?:Li(\d)E)?\S*'.*?Used (\d+) registers", p.stderr, re.S)
    kernels = {(mode, blocks): int(n) for mode, blocks, n in found}
    assert kernels["1", "3"] <= 80 and kernels["0", "3"] <= 80 and kernels["0", "1"] <= 168, kernels
