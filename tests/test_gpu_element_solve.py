"""The element solve keeps every right-hand side's own precision, however large its element's others are."""
import numpy as np
import pytest

from paper_2402_04514_gb300 import assembly


@pytest.mark.gpu
@pytest.mark.parametrize("small", [1e-9, 1e-20])
def test_lumped_mass_keeps_small_changes(small):
    """With a diagonal M_K, d^H = d^L (c_ev so large that every indicator saturates) and no limiter, U^H is U^L.  The
    right-hand sides of m_y are of order 1 at the nodes that face the jump in m_y and of order `small` at the other nodes
    of the same elements; each must come out to its own rounding: of U, and of the few products that dU is made of."""
    import copy

    import torch

    from paper_2402_04514_gb300.gdg import Solver

    P = copy.copy(assembly.assemble_2d(8, 6, 1))
    nl = P.n_loc
    P.MK = np.zeros_like(P.MK)
    for a in range(nl):
        P.MK[:, a, a] = P.mi.reshape(-1, nl)[:, a]
    left = np.repeat(P.x[0].reshape(-1, nl).mean(1) < 0.5, nl)
    my = np.where(left, 1.0, small * np.random.default_rng(3).uniform(1, 2, P.n))
    U = np.stack([np.ones(P.n), np.full(P.n, 0.5), my, np.where(left, 3.125, 2.625)])
    Ud = torch.from_numpy(U).cuda()
    out = []
    for order in (0, 1):  # low, high
        S = Solver(P, params=dict(order=order, c_ev=1e300))
        out.append(S.stage(Ud, 1e-3).cpu().numpy())
    dU = np.abs(out[0] - U)
    assert dU[2][~left].max() > 1e-3  # the jump's nodes
    assert (np.abs(out[1] - out[0]) <= 4 * 2.0 ** -52 * (np.abs(U) + dU)).all()
