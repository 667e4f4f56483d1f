"""The density limit of the line searches is a correctly rounded quotient, as the closed form states it."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("approx", [None, "((y)*(1.0-6.8e-8))", "((y)*(1.0+6.8e-8))"])
def test_integer_quotient(tmp_path, approx):
    """csrc/fixfp64.cuh as host C++ against the processor's division, its starting approximation moved to both ends of the
    instruction's documented error too."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "check")
    hook = [] if approx is None else ["-DSF_HOST_APPROX(y)=" + approx]
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", *hook, os.path.join(HERE, "quot_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe, "4000000", "1"], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr


@pytest.mark.gpu
def test_density_limited_factors():
    """Where the density bounds alone limit an entry, its factor is the quotient's own bits in the row that limits it."""
    import torch

    from oracle.oracle import Oracle
    from paper_2402_04514_gb300.gdg import Solver
    from tests.helpers import four_quadrant_problem

    P, U = four_quadrant_problem(24, 2, seed=4)
    O, S = Oracle(P), Solver(P)
    tau = O.max_dt(U, 0.5)
    for _ in range(6):
        U = O.stage(U, tau)[0]
    S.stage(torch.from_numpy(U).cuda(), tau)
    UL, A, rmin, rmax, l1 = (S.export(k) for k in ("UL", "A", "rho_min", "rho_max", "l1"))
    rows, col = np.repeat(np.arange(P.n), np.diff(P.row_ptr)), P.col_idx
    rho, a = UL.reshape(4, -1)[0], A.reshape(4, -1)[0]
    w = (np.diff(P.row_ptr) + np.bincount(P.b_node, minlength=P.n)) / P.mi

    def limit(i, pr):
        r1 = rho[i] + pr
        with np.errstate(all="ignore"):
            l = np.where(r1 < rmin[i], (rmin[i] - rho[i]) / pr, 1.0)
            l = np.where(r1 > rmax[i], (rmax[i] - rho[i]) / pr, l)
        return np.clip(l, 0.0, 1.0)

    want = np.minimum(limit(rows, w[rows] * a), limit(col, w[col] * -a))
    near = (want < 1.0) & (want > 0.0) & (np.abs(l1 - want) <= 4 * np.spacing(want))  # the others psi limits further
    assert near.sum() > 500
    assert (l1[near] == want[near]).all()
