"""Algorithmic work of each sweep kernel per launch: compulsory HBM bytes and FP64 operations.

Bytes: every array a kernel must read is read once and every array it writes is written once (per-entry
arrays of nnz entries, per-node arrays of n nodes); neighbour states are counted once per node, not per
entry (an ideal cache), and what a kernel reads back of its own output is not counted.  FP64 operations: the
arithmetic as the kernels state it for states of which no two agree, counted per undirected edge, per stencil
entry (c_ij != 0), per pair of nodes of an element, per node and per boundary entry, with add/sub/mul = 1, fused
multiply-add = 2, and division, square root and power = 1 each (the usual floating-point operation count; their
cost in hardware is several to ~100 FMA issue slots, which is why the sweep is bound by arithmetic: the FP64 pipe
and, for the products the kernels move there, the integer pipe).  FP32 work (the line searches' certificates) is not
counted, nor what depends on the data: the deferred line searches, and the second pass of rows with a
remainder, so that the FP64 fraction reported is a lower bound.
"""
from __future__ import annotations

from dataclasses import dataclass

import numpy as np

KERNELS = ("prim", "maxdt", "low", "high", "limit2", "final", "edge", "lsfix", "tau", "clock", "axpy")


@dataclass
class Counts:
    dim: int
    n: int
    nnz: int  # CSR entries
    nnz_s: int  # entries with c_ij != 0
    nb: int
    n_loc: int

    @property
    def m(self):
        return self.dim + 2

    @staticmethod
    def of(problem):
        cs = np.abs(problem.cij).sum(0) > 0
        return Counts(problem.dim, int(problem.n), int(problem.col_idx.size), int(cs.sum()), int(problem.b_node.size),
                      int(problem.n_loc))


def bytes_per_launch(c: Counts) -> dict:
    m, d, n, nnz, s, nb, nl = c.m, c.dim, c.n, c.nnz, c.nnz_s, c.nb, c.n_loc
    edge_geom = (s // 2) * (4 * 4 + 8 * (1 + d))  # entry, row, column, transpose; |c| and n_ij of one of the two entries
    side_geom = nb * (3 * 4 + 8 * (1 + d))  # node, type, caller's index; |c| and normal of a boundary entry
    pairs = n * (nl - 1) // 2  # of nodes of one element
    return dict(
        prim=8 * n * (m + m + 7),  # U -> U by slots, seven primitives
        maxdt=edge_geom + 8 * n * (d + 5) + 8 * s + side_geom + 8 * nb,
        # d, G, the indicator's term, rho and s~ of the bar state at both entries; a boundary entry's state, two
        # fluxes, d and bar state
        edge=edge_geom + 8 * n * (m + 7) + 8 * s * (m + 4) + side_geom + 8 * nb * (3 * m + 3),
        low=n * 12 + 8 * n * (m + 4 + 1) + s * (4 + 8 * (m + 4)) + 8 * n * (2 * m + 4) + 8 * nb * (3 * m + 1),
        # the rows' states, right-hand sides, U^L, aggregates, bounds, N and factors of the bounds and of P; M_K^-1;
        # column, d, mu of the stencil; m_ij and transpose of an element's pairs; A and the factors
        high=n * 17 + 8 * n * (3 * m + 3 + 3 + 1 + 2 + 1) + 8 * n * nl + 4 * nnz + 16 * s + 12 * pairs + 8 * nnz * (m + 1)
        + 8 * nb * (2 * m + 5),
        limit2=n * 14 + 8 * n * (2 * m + 1) + nnz * (4 + 8 * (m + 1)) + 8 * nb * (m + 1),
        final=8 * m * n * 3 + n,
        lsfix=0,  # the deferred line searches: data-dependent, not counted
        tau=n * (12 + 8) + 8 * s + 8 * nb,
        clock=0,
        axpy=8 * m * n * 3,
    )


def quiet_bytes_per_launch(c: Counts) -> dict:
    """bytes_per_launch of a mesh on which every state is the same: the edge sweep stores d_ij alone, sweep A reads nothing else
    of an entry but its column, the element sweep writes bounds and factors but no A, and sweep C reads no entry."""
    m, n, nnz, s, nb = c.m, c.n, c.nnz, c.nnz_s, c.nb
    out = bytes_per_launch(c)
    out["edge"] -= 8 * s * (m + 3)
    out["low"] -= 8 * s * (m + 3)
    out["high"] = n * 17 + 8 * n * (2 * m + 3 + 3 + 1 + 2) + 4 * s + 8 * nnz + 8 * nb * (2 * m + 5)
    out["limit2"] = n * 14 + 8 * n * (2 * m + 1) + 8 * nb * (m + 1)
    return out


def flops_per_launch(c: Counts) -> dict:
    m, d, n, s, nb, nl = c.m, c.dim, c.n, c.nnz_s, c.nb, c.n_loc
    pairs = n * (nl - 1) // 2
    lam = 23  # wave-speed bound from the stored primitives
    vel = 4 * d  # two normal momenta and velocities
    flux = 2 * (3 * d + 2)  # f(U_i) n and f(U_j) n
    edge_pair = vel + lam + 1 + d + 4 + flux + 1 + 4 * m + 3 + (2 * d + 7)  # d_ij, G, W, the indicator's term, s~ of the bar state
    side = 4 * d + 1 + (2 * d + 3) + vel + 5 + lam + 1  # a boundary entry's state, its primitives and d
    low_node = 4 + 1 + 4 * m + (2 + d + 2 * d - 1 + 6 + 3 * d + 2) + 4 * m + 2
    return dict(
        edge=(s // 2) * edge_pair + nb * (side + flux + 3 + 7 * m + 2 * d + 5),
        prim=n * (2 * d + 13),
        maxdt=(s // 2) * (vel + lam + 1) + nb * side,
        low=s * (4 * m + 2) + n * low_node + nb * (5 * m + 1),
        high=s * (4 * m + 5) + pairs * 3 * m + n * (2 * nl * m + m + 3 + (2 * d + 8)) + nb * (5 * m + 3),
        limit2=c.nnz * 2 * m + n * 2 * m + nb * 2 * m,
        final=n * 3 * m,
        lsfix=0,
        tau=s + 3 * n + nb,
        clock=0,
        axpy=3 * m * n,
    )


# FP64 pipe peak from unit counts and clocks: 152 SMs x 2 FP64 FMA per clock per SM x 2 flop x 2.07 GHz.
FP64_PEAK_TFLOPS = 152 * 2 * 2 * 2.07e9 / 1e12
# The sweep kernels also run binary64 products on the integer pipe (csrc/softfp64.cuh).  One such product
# issues INT_MUL_ALU_INST instructions on the ALU pipe (ncu instruction counts of a kernel doing nothing
# else; the rest go to the FMA-heavy pipe, which is not the tighter one), and the ALU pipe retires 64
# thread-instructions per clock per SM, so the integer pipes add 64 / INT_MUL_ALU_INST products (1 flop each)
# per clock per SM.  The arithmetic roof of a kernel that keeps both pipes busy is the sum of the two.
INT_MUL_ALU_INST = 33
INT_MUL_PEAK_TFLOPS = 152 * 64 / INT_MUL_ALU_INST * 2.07e9 / 1e12
ALU_PEAK_TFLOPS = FP64_PEAK_TFLOPS + INT_MUL_PEAK_TFLOPS


def library_source_digest() -> str:
    """sha256 (first 16 hex digits) of the library's CUDA sources and public header.  A DRAM-traffic figure
    taken with ncu is only valid for the sources it was taken from; bench.py reports it only while this
    digest matches the one recorded beside the figure."""
    import glob
    import hashlib
    import os

    here = os.path.dirname(os.path.abspath(__file__))
    files = sorted(glob.glob(os.path.join(here, "csrc", "*.cu")) + glob.glob(os.path.join(here, "csrc", "*.cuh")))
    files.append(os.path.join(os.path.dirname(here), "include", "gdg.h"))
    h = hashlib.sha256()
    for f in files:
        h.update(os.path.basename(f).encode())
        with open(f, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def measured_traffic(path: str, kernel: str, n_nodes: int, precision: str = "fp64"):
    """DRAM bytes (read + write) per launch of `kernel` from an ncu summary table (lines
    `kernel nodes dram_read_bytes dram_write_bytes source_digest [precision]`, precision fp64 when absent),
    scaled from the captured mesh to `n_nodes` (every array a sweep kernel touches grows in proportion to
    the node count).  None when the table is missing, has no row for the kernel and precision, or was
    taken from other sources."""
    try:
        with open(path) as fh:
            lines = [ln.split() for ln in fh if ln.strip() and not ln.lstrip().startswith("#")]
    except OSError:
        return None
    digest = library_source_digest()
    for f in lines:
        if len(f) in (5, 6) and f[0] == kernel and f[4] == digest and (f[5] if len(f) == 6 else "fp64") == precision:
            return (float(f[2]) + float(f[3])) * n_nodes / float(f[1])
    return None
