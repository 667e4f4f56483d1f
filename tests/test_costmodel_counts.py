"""The work model counts what the kernels do: per entry, pair, node and boundary entry, read off by differences."""
from paper_2402_04514_gb300 import costmodel
from paper_2402_04514_gb300.costmodel import Counts


def _per(fn, kernel, **one):
    """The model's slope in one of its counts, on a large mesh of Q2 quads."""
    base = dict(dim=2, n=9000, nnz=140000, nnz_s=130000, nb=600, n_loc=9)
    more = {k: base[k] + 1000 * v for k, v in one.items()}
    return (fn(Counts(**{**base, **more}))[kernel] - fn(Counts(**base))[kernel]) / 1000


def test_operations_of_q2_quads():
    f = costmodel.flops_per_launch
    # the edge sweep, per undirected edge: two normal velocities 8, lambda 23 and d 1, c 2 and its products 4, two fluxes 16, 1 / d 1,
    # differences and bar state 16, indicator 3, s~ of the bar state 11
    assert _per(f, "edge", nnz_s=2) == 85
    assert _per(f, "maxdt", nnz_s=2) == 32  # one thread per edge
    assert _per(f, "low", nnz_s=1) == 18  # 14 instructions, four of them fused multiply-adds
    assert _per(f, "high", nnz_s=1) == 21  # no evaluation of psi in the sweep
    assert _per(f, "high", nnz=1) == 0
    assert _per(f, "high", n=1) == 72 + 4 + 3 + 12 + 4 * 12  # the element solve, bounds, the row's search context, four pairs
    assert _per(f, "limit2", nnz=1) == 8
    assert _per(f, "tau", nnz_s=1) == 1 and _per(f, "tau", nb=1) == 1  # boundary wave speeds belong to the edge sweep
    assert _per(f, "edge", nb=1) == 18 * 2 + 45 + 7 * 4 and _per(f, "low", nb=1) == 21


def test_bytes_of_q2_quads():
    b, q = costmodel.bytes_per_launch, costmodel.quiet_bytes_per_launch
    assert _per(b, "low", nnz_s=1) == 4 + 8 * 8  # column; d, G (4), indicator term, rho and s~ of the bar state, once per entry
    assert _per(b, "edge", nnz_s=2) == 16 + 24 + 2 * 8 * 8
    assert _per(b, "high", nnz=1) == 4 + 8 * 5 and _per(b, "high", nnz_s=1) == 16
    assert _per(q, "low", nnz_s=1) == 12 and _per(q, "edge", nnz_s=2) == 56 and _per(q, "high", nnz=1) == 8
    for k in ("edge", "low", "high", "limit2"):
        c = Counts(dim=2, n=9000, nnz=140000, nnz_s=130000, nb=600, n_loc=9)
        assert 0 < q(c)[k] < b(c)[k]
