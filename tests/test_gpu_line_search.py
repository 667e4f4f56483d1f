"""The deferred line searches (k_lsfix): FP32 root, Newton steps in FP64, bracketed iteration where those do not settle."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2402_04514_gb300 import assembly, workloads
from paper_2402_04514_gb300.gdg import Solver
from tests.helpers import dirichlet_vortex_problem, four_quadrant_problem, octant_problem

pytestmark = pytest.mark.gpu


def _case(name):
    if name == "sod_q1":
        P = assembly.assemble_1d(60, 1)
        return P, workloads.sod(P.x[0]), None, 1.4
    if name == "vortex_q3_gamma53":
        P, U, bd = dirichlet_vortex_problem(12, 3)
        return P, U, np.ascontiguousarray(bd(0.0)), 5.0 / 3.0
    if name == "quadrants_q2_gamma_general":  # a gamma that is no ratio with a small denominator
        P, U = four_quadrant_problem(13, 2, seed=4, gamma=1.37123)
        return P, U, None, 1.37123
    P, U = octant_problem((6, 5, 7), 1, seed=2) if name == "octants_q1" else octant_problem((3, 4, 3), 2, seed=2)
    return P, U, None, 1.4


@pytest.mark.parametrize("name", ["sod_q1", "vortex_q3_gamma53", "quadrants_q2_gamma_general", "octants_q1", "octants_q2"])
def test_factors_against_oracle(name):
    """l of both passes after seven stages.  Where the search iterates, its end is the root of psi to the tolerance 1e-14
    plus what psi's own rounding leaves open: a few ulp of E over |psi'| in row i or row j (l is their minimum); 16 ulp cover
    both evaluations.  The second factor also moves with the first ones, each known to its own tolerance t: by l2 t / (1 - l1)
    through the entry's remainder, and through the row's U^(1) by the sum of t |grad psi . A| / m over the row, over |psi'|."""
    import torch

    P, U, B, gamma = _case(name)
    S, O = Solver(P, gamma), Oracle(P, gamma=gamma)
    kw = {} if B is None else dict(bdata=B)
    Bd = None if B is None else torch.from_numpy(B).cuda()
    tau = O.max_dt(U, 0.5, **kw)
    for _ in range(6):  # the flow after six stages: limiter active around the fronts
        U = O.stage(U, tau, **kw)[0]
    S.stage(torch.from_numpy(U).cuda(), tau, bdata=Bd)
    _, _, tr = O.stage(U, tau, trace=True, **kw)
    assert P.dim == 1 or S.export("ls_deferred").sum() > 0
    rows = np.repeat(np.arange(P.n), np.diff(P.row_ptr))
    ikm = (np.diff(P.row_ptr) + np.bincount(P.b_node, minlength=P.n)) / P.mi
    for k, U0, w in (("l1", tr["UL"], np.ones(P.nnz)), ("l2", tr["U1"], 1.0 - tr["l1"])):
        l, ref = S.export(k), tr[k]
        on = np.ones(P.nnz, bool) if k == "l1" else (S.export("l1") < 1.0) & (tr["l1"] < 1.0)
        slope, more = np.full(P.nnz, np.inf), np.zeros(P.nnz)
        for r in (rows, P.col_idx):  # |d psi / d l| from either row's side
            q = (1.0 if r is rows else -1.0) * w * ikm[r] * tr["A"]
            V = U0[:, r] + ref * q
            m2 = (V[1:-1] ** 2).sum(0)
            d = q[-1] - (V[1:-1] * q[1:-1]).sum(0) / V[0] + 0.5 * m2 * q[0] / V[0] ** 2 \
                - tr["s_min"][r] * gamma * V[0] ** (gamma - 1) * q[0]
            slope = np.minimum(slope, np.abs(d) / V[-1])
            if k == "l2":
                v = U0[1:-1] / U0[0]
                grad = np.concatenate([[0.5 * (v * v).sum(0) - tr["s_min"] * gamma * U0[0] ** (gamma - 1)], -v, np.ones((1, P.n))])
                moved = np.bincount(rows, (tr["l1"] < 1.0) * tol * np.abs((grad[:, rows] * tr["A"]).sum(0)), minlength=P.n) / P.mi
                more = np.maximum(more, moved[r] / np.maximum(np.abs(d), 1e-300))
        if k == "l2":
            more += ref * tol / np.maximum(1.0 - tr["l1"], 1e-300)
        tol = 1e-14 + 16 * 2.2e-16 / np.maximum(slope, 1e-300) + more
        assert (np.abs(l - ref)[on] <= np.minimum(tol, 1.0)[on]).all(), (k, np.abs(l - ref)[on].max())
