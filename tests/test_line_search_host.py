"""The deferred line searches, compiled as host C++ and run on the searches that the oracle's limiter passes pose."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2402_04514_gb300 import assembly, workloads
from tests.helpers import dirichlet_vortex_problem, four_quadrant_problem, octant_problem

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def _case(name):
    if name == "sod_q1":
        P = assembly.assemble_1d(60, 1)
        return P, workloads.sod(P.x[0]), None, 1.4
    if name == "vortex_q3":
        P, U, bd = dirichlet_vortex_problem(12, 3)
        return P, U, np.ascontiguousarray(bd(0.0)), 5.0 / 3.0
    if name == "quadrants_q2":
        P, U = four_quadrant_problem(24, 2, seed=4)
        return P, U, None, 1.4
    P, U = octant_problem((8, 7, 6), 1, seed=2)
    return P, U, None, 1.4


@pytest.mark.skipif(np.finfo(np.longdouble).eps > 1e-18, reason="no long double wider than double")
@pytest.mark.parametrize("name", ["sod_q1", "vortex_q3", "quadrants_q2", "octants_q1"])
def test_line_search_ends_at_the_rounding_of_psi(tmp_path, name):
    """Half of what the tolerance and psi's rounding leave open, in the root mean square: the bracketed iteration alone is at
    0.21 to 0.27 of it."""
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    P, U, B, gamma = _case(name)
    O, kw = Oracle(P, gamma=gamma), {} if B is None else dict(bdata=B)
    tau = O.max_dt(U, 0.5, **kw)
    rows = np.repeat(np.arange(P.n), np.diff(P.row_ptr))
    ikm = (np.diff(P.row_ptr) + np.bincount(P.b_node, minlength=P.n)) / P.mi
    recs = []
    for s in range(9):
        U, _, tr = O.stage(U, tau, trace=True, **kw)
        i = np.nonzero(tr["l1"] < 1.0)[0]
        r = rows[i]
        for U0, w in ((tr["UL"], ikm[r]), (tr["U1"], (1.0 - tr["l1"][i]) * ikm[r])):
            if s >= 5:
                recs.append(np.vstack([U0[:, r], tr["A"][:, i], w, tr["rho_min"][r], tr["rho_max"][r], tr["s_min"][r]]).T)
    R = np.ascontiguousarray(np.concatenate(recs))
    data, exe = str(tmp_path / "searches"), str(tmp_path / "check")
    np.concatenate([[P.dim, gamma, R.shape[0]], R.ravel()]).tofile(data)
    subprocess.run([cxx, "-O2", "-std=c++17", "-w", "-ffp-contract=off", "-I" + os.path.join(CUDA, "include"),
                    os.path.join(HERE, "line_search_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe, data], capture_output=True, text=True)
    print(out.stdout)
    assert out.returncode == 0, out.stdout + out.stderr


def test_flat_directions_are_not_given_up(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path / "check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-w", "-ffp-contract=off", "-I" + os.path.join(CUDA, "include"),
                    os.path.join(HERE, "flat_search_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    print(out.stdout)
    assert out.returncode == 0, out.stdout + out.stderr
