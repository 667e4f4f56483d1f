"""The time-step bound of gdg_max_dt and of a fused step's first stage are the same bits, boundary entries included."""
import numpy as np
import pytest

from paper_2402_04514_gb300 import assembly, workloads
from tests.helpers import inoutflow_case, octant_problem

pytestmark = pytest.mark.gpu


def _case(name, rng):
    """A random state, so that no two entries agree, with boundary data that is faster than the interior: the bound is taken
    at a boundary node."""
    if name == "slip_q2":
        P = assembly.assemble_2d(9, 7, 2)
    elif name == "dirichlet_q3":
        P = assembly.assemble_2d(5, 6, 3, bc=dict(left="dirichlet", right="dirichlet", bottom="dirichlet", top="slip"))
    elif name == "octants":
        P = octant_problem((4, 5, 3), 1, seed=1, bc=dict(left="inoutflow", right="dirichlet"))[0]
    else:
        P = inoutflow_case(name)[0]

    def state(n, fast):
        rho, p, v = rng.uniform(0.5, 2, n), rng.uniform(0.5, 2, n), rng.uniform(-0.2, 0.2, (P.dim, n))
        return workloads.prim_to_cons(rho, fast * v, fast * fast * p, 1.4)

    return P, state(P.n, 1.0), np.ascontiguousarray(state(P.nb, 3.0))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", ["slip_q2", "dirichlet_q3", "octants", "sod1d_open", "fq_q2_open_sides"])
def test_same_bits_as_the_fused_step(name, precision):
    import torch

    from paper_2402_04514_gb300.gdg import Solver

    for seed in range(8):
        P, U, B = _case(name, np.random.default_rng(seed))
        S = Solver(P, params=dict(precision=precision))
        Ud, Bd = torch.from_numpy(U).cuda(), torch.from_numpy(B).cuda()
        tau = S.max_dt(Ud, 0.5, bdata=Bd)
        S.set_clock(0.0, float("inf"), 0.5)
        S.step(Ud, (torch.empty_like(Ud), torch.empty_like(Ud)), bdata=Bd)
        assert S.clock()[1] == tau, (seed, S.clock()[1], tau)
