"""The element solve's fixed-point dot products (csrc/fixfp64.cuh), compiled as host C++, over the inverse element masses of every
element the library's meshes have: no further from long double than the FP64 sums, in the mean square and within a bound."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2402_04514_gb300 import assembly

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 1e-18, reason="no long double wider than double")
@pytest.mark.parametrize("dim,degree", [(1, 1), (1, 3), (2, 1), (2, 2), (2, 3), (3, 1), (3, 2)])
def test_fixed_point_dot(tmp_path, dim, degree):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    P = {1: lambda: assembly.assemble_1d(5, degree), 2: lambda: assembly.assemble_2d(3, 5, degree),
         3: lambda: assembly.assemble_3d(3, 2, 4, degree)}[dim]()
    W = np.linalg.inv(P.MK[0])
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", os.path.join(HERE, "fixdot_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe, "20000", "3"], input="%d\n%s" % (W.shape[0], " ".join(float(v).hex() for v in W.ravel())),
                         capture_output=True, text=True)
    print(out.stdout)
    assert out.returncode == 0, out.stdout + out.stderr
