"""The integer-pipe reciprocal, square root and inverse roots (csrc/fixfp64.cuh) over all that their starting approximations may
be: on the host with the approximations moved to the ends of the instructions' documented errors, on the GPU over every
FP32 significand."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 1e-18, reason="no long double wider than double")
@pytest.mark.parametrize("sign", ["-", "+"])
def test_approximations_at_the_ends_of_their_errors(tmp_path, sign):
    """rcp.approx and rsqrt.approx are documented to 2^-23 and 2^-22.9 = 1.27e-7 of the value, of which rounding to FP32 may
    take 2^-24: the rest is put on the value before that rounding.  Below 1/2 it leaves the binade that the exact value is in."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-DSF_HOST_APPROX(y)=((y)*(1.0%s6.8e-8))" % sign,
                    os.path.join(HERE, "fixfp64_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe, "500000", "2"], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr


@pytest.mark.gpu
def test_every_starting_significand():
    """Every FP32 significand the approximations start from, at both parities of the exponent, with the lowest and the highest
    bits below it: within 9/16 ulp of the exact value, so one step from CUDA's correctly rounded results at most."""
    torch = pytest.importorskip("torch")
    from paper_2402_04514_gb300.gdg import math_selftest

    top = torch.arange(1 << 23, dtype=torch.int64, device="cuda") << 29
    for low in (0, (1 << 29) - 1):
        for field in (1023, 1024):
            x = ((field << 52) | top | low).view(torch.float64)
            for mine, ref in ((0, 2), (5, 6)):
                d = (math_selftest(mine, 1, x).view(torch.int64) - math_selftest(ref, 1, x).view(torch.int64)).abs()
                assert int(d.max()) <= 1, (mine, field, low)
