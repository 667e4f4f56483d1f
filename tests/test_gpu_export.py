"""What gdg_debug_export gives between and after calls that do not work everything out."""
import numpy as np
import pytest

from paper_2402_04514_gb300 import assembly, workloads
from paper_2402_04514_gb300.gdg import Solver

pytestmark = pytest.mark.gpu

NAMES = ("dL", "dB", "N", "UL", "U1", "A", "rho_min", "rho_max", "s_min", "l1", "l2")


@pytest.mark.parametrize("dim,degree", [(1, 1), (2, 2), (3, 1)])
def test_time_step_query_leaves_the_last_stage(dim, degree):
    import torch

    P = {1: lambda: assembly.assemble_1d(37, degree), 2: lambda: assembly.assemble_2d(9, 7, degree),
         3: lambda: assembly.assemble_3d(3, 5, 4, degree)}[dim]()
    rng = np.random.default_rng(1)
    U = np.zeros((dim + 2, P.n))
    U[0], U[1:-1], U[-1] = rng.uniform(1, 2, P.n), rng.uniform(-0.3, 0.3, (dim, P.n)), rng.uniform(3, 5, P.n)
    S = Solver(P)
    Ud, Vd = torch.from_numpy(U).cuda(), torch.from_numpy(U[:, ::-1].copy()).cuda()
    S.stage(Ud, S.max_dt(Ud, 0.4))
    before = {k: S.export(k) for k in NAMES}
    S.max_dt(Vd, 0.4)
    for k in NAMES:
        assert np.array_equal(S.export(k), before[k], equal_nan=True), k


def test_unlimited_stage_exports_zeros_between_equal_states():
    """A after a stage of order HIGH that follows one of another state: zero wherever the two states are equal."""
    import torch

    P = assembly.assemble_2d(12, 11, 2)
    rng = np.random.default_rng(2)
    U = np.stack([rng.uniform(1, 2, P.n), rng.uniform(-0.3, 0.3, P.n), rng.uniform(-0.3, 0.3, P.n), rng.uniform(3, 5, P.n)])
    V = workloads.four_quadrant(P.x[0], P.x[1], seed=3)
    S = Solver(P)
    S.stage(torch.from_numpy(U).cuda(), 1e-4)
    S.set_params(order=1)
    S.stage(torch.from_numpy(V).cuda(), 1e-4)
    A = S.export("A").reshape(4, -1)
    rows = np.repeat(np.arange(P.n), np.diff(P.row_ptr))
    equal = (V[:, rows] == V[:, P.col_idx]).all(0) & (np.abs(P.cij).max(0) > 0)
    assert equal.sum() > 1000 and (A[:, equal] == 0).all()
