"""The integer-pipe reciprocal, square root, inverse roots and unpacked products (csrc/fixfp64.cuh), the header compiled as host C++
against long double: within one rounding (plus 1/16 ulp) of the exact value.  On the GPU, whose approximations they start from,
test_gpu_parity.py compares them with CUDA's operations."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 1e-18, reason="no long double wider than double")
@pytest.mark.parametrize("seed", [0, 1])
def test_fixed_point_functions(tmp_path, seed):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", os.path.join(HERE, "fixfp64_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe, "1000000", str(seed)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
