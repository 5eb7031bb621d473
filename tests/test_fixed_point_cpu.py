"""The integer arithmetic of the FP64 path (esdg_fixed.cuh), compiled for the host."""

import os
import shutil
import subprocess

import pytest

from paper_2005_02516_gb300 import _build


def _run(tmp_path, program):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no CUDA compiler")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text('#include "esdg_fixed.cuh"\n#include <cmath>\n#include <cstdio>\n#include <cstdlib>\n#include <random>\n'
                   "using namespace esdg;\n#define CHECK(c) if (!(c)) { printf(\"line %d: %s\\n\", __LINE__, #c); return 1; }\n"
                   + program)
    subprocess.run([_build.nvcc(), "-std=c++17", "-O1", *_build.ARCH, "-I", _build.CSRC, str(src), "-o", str(exe)],
                   check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert p.returncode == 0, p.stdout


def test_larger_speed_keeps_a_nan_of_either_sign(tmp_path):
    _run(tmp_path, r"""
int main() {
    const double nan = fx_double(0x7ff8000000000000ll), minus_nan = fx_double((long long)0xfff8000000000000ull);
    for (double n : {nan, minus_nan})
        for (double x : {0.0, 1.0, HUGE_VAL, 5e-324}) {
            CHECK(std::isnan(r_max_nonneg(n, x)));
            CHECK(std::isnan(r_max_nonneg(x, n)));
        }
    const double v[] = {0.0, 5e-324, 1e-300, 0.5, 1.0, 1.0 + 0x1p-52, 1e300, HUGE_VAL};
    for (double a : v)
        for (double b : v) CHECK(r_max_nonneg(a, b) == (a > b ? a : b));
    return 0;
}
""")
