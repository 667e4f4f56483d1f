"""Equal states: entries between them are skipped by the edge sweep and both row sweeps, and a row whose antidiffusive fluxes
are all zero is marked instead of written.  A wave on a constant background, so that quiet rows, quiet rows in active elements,
active rows with some equal neighbours and boundary rows all occur, and the wave then runs over rows that held other data."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2402_04514_gb300 import assembly, gdg
from paper_2402_04514_gb300.gdg import Solver

pytestmark = pytest.mark.gpu

CASES = [(1, 1, (70,)), (1, 3, (40,)), (2, 1, (34, 9)), (2, 2, (17, 13)), (2, 3, (9, 7)), (3, 1, (7, 6, 5)), (3, 2, (4, 3, 3))]


def _problem(dim, degree, ns, periodic):
    make = (assembly.assemble_1d, assembly.assemble_2d, assembly.assemble_3d)[dim - 1]
    box = (0.0, 1.0) * dim
    P = make(ns[0], degree, 0.0, 1.0, periodic=periodic) if dim == 1 else make(*ns, degree, box=box, periodic=(periodic,) * dim)
    rho = np.where((P.x < 0.3).all(0), 1.0, 0.4)
    U = np.zeros((dim + 2, P.n))
    U[0], U[1], U[-1] = rho, 0.3 * rho, 2.5 * np.where((P.x < 0.3).all(0), 1.0, 0.3) + 0.045 * rho
    return P, U


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("dim,degree,ns", CASES)
def test_wave_on_a_constant_state(dim, degree, ns, periodic):
    """Five stages on the same handle against the oracle from the same inputs, 1e-12 of each component's largest value (as the
    parity tests of the stage); in between a stage of smooth data, which leaves nothing equal and other numbers in the scratch."""
    import torch

    P, U = _problem(dim, degree, ns, periodic)
    S, O = Solver(P), Oracle(P)
    tau = O.max_dt(U, 0.5)
    assert abs(S.max_dt(torch.from_numpy(U).cuda(), 0.5) - tau) <= 1e-13 * tau
    smooth = U * (1.0 + 0.01 * np.sin(7.0 * P.x.sum(0) + 0.3))
    for k in range(5):
        if k == 2:
            S.stage(torch.from_numpy(smooth).cuda(), 0.3 * tau)
        out = S.stage(torch.from_numpy(U).cuda(), tau).cpu().numpy()
        ref, flags, tr = O.stage(U, tau, trace=True)
        for q in range(dim + 2):
            assert np.abs(out[q] - ref[q]).max() <= 1e-12 * max(np.abs(ref[q]).max(), 1e-3), (k, q)
        A, l1 = S.export("A").reshape(tr["A"].shape), S.export("l1")
        assert np.abs(A - tr["A"]).max() <= 1e-12 * np.abs(tr["A"]).max()
        on = ((tr["A"] == 0.0) & (A == 0.0)).all(0)  # no flux: the factor is 1
        assert (l1[on] == 1.0).all() and (on.any() or k > 2)
        assert flags == 0 and S.status() == 0
        U = ref


def test_uniform_state_is_kept():
    """One state everywhere, periodic: every pass skips every entry, and the state comes back bit for bit; the same for mixed."""
    import torch

    P = assembly.assemble_2d(33, 18, 2, periodic=(True, True))
    U = np.tile(np.array([0.7, 0.2, -0.4, 1.9])[:, None], (1, P.n))
    for precision in (gdg.PRECISION_FP64, gdg.PRECISION_MIXED):
        S = Solver(P, 1.4, dict(precision=precision))
        Ud = torch.from_numpy(U).cuda()
        tau = S.max_dt(Ud, 0.5)
        assert np.isfinite(tau)
        assert (S.stage(Ud, tau).cpu().numpy() == U).all() and S.status() == 0
        assert (S.export("A") == 0.0).all() and (S.export("l1") == 1.0).all()
