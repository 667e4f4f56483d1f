"""The sweeps' instantiations for full launches (tighter register caps, gdg_internal.cuh: few_threads) as single instances: one stage of
meshes just above the threshold, 116,736 threads, against the oracle."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2402_04514_gb300 import assembly, workloads
from tests.helpers import octant_problem, rel_err

pytestmark = pytest.mark.gpu

FULL = 152 * 768
CASES = {
    "1d_q1": (1, (59000,), 1, {}), "1d_q3": (1, (30000,), 3, {}),
    "2d_q1_open": (2, (173, 171), 1, dict(left="inoutflow", right="inoutflow", bottom="inoutflow", top="inoutflow")),
    "2d_q2": (2, (115, 114), 2, {}), "2d_q3_dirichlet": (2, (87, 86), 3, dict(left="dirichlet", right="dirichlet")),
    "3d_q1": (3, (26, 25, 24), 1, {}), "3d_q2_open": (3, (17, 17, 16), 2, dict(left="inoutflow", right="inoutflow")),
}


def _build(name):
    dim, cells, degree, bc = CASES[name]
    if dim == 1:
        P = assembly.assemble_1d(*cells, degree)
        U = workloads.sod(P.x[0])
    elif dim == 2:
        P = assembly.assemble_2d(*cells, degree, bc=bc) if bc else assembly.assemble_2d(*cells, degree)
        U = workloads.four_quadrant(P.x[0], P.x[1], seed=2)
    else:
        P, U = octant_problem(cells, degree, seed=2, bc=bc or None)
    wave = 1 + 0.05 * np.sin(9 * P.x[0] + (7 * P.x[-1] if dim > 1 else 0))  # no two nodes equal beside the jumps
    return P, U * wave, np.ascontiguousarray((U * wave)[:, P.b_node])


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("what", ["limited", "low", "high", "mixed"])
def test_stage_against_oracle(name, what):
    """1e-12 of the component's largest value, as the small meshes' stages; mixed 2e-5 (test_gpu_mixed)."""
    import torch

    from paper_2402_04514_gb300.gdg import Solver

    P, U, B = _build(name)
    assert -(-P.n // (32 * P.n_loc)) * 32 * P.n_loc > FULL
    order, mixed = dict(limited=2, low=0, high=1, mixed=2)[what], what == "mixed"
    O, S = Oracle(P, params=dict(order=order), openmp=True), Solver(P, params=dict(order=order, precision=int(mixed)))
    tau = O.max_dt(U, 0.3, bdata=B)
    ref, flags = O.stage(U, tau, bdata=B)
    out = S.stage(torch.from_numpy(U).cuda(), tau, bdata=torch.from_numpy(B).cuda()).cpu().numpy()
    assert rel_err(out, ref) <= (2e-5 if mixed else 1e-12) and S.status() == flags == 0
