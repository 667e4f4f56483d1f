// Sweep B: high-order update with the consistent element mass, relaxed local bounds, antidiffusive
// fluxes and the first convex-limiting pass.  One thread per node; a block holds whole elements so the
// element solve and the m_ij coupling of A_ij stay in shared memory.
#include <type_traits>

#include "gdg_internal.cuh"

namespace gdg {

namespace {

constexpr int kMaxBlock = kHighMaxBlock;
constexpr int kMaxLocal = 32;  // n_loc limit of gdg_setup

// Thread-to-node map of an element block.  A block holds eb elements (a power of two <= kEll) of one
// ELL group of kEll consecutive elements: block lb of an instance takes group g = lb / (kEll / eb) and its
// elements e0 .. e0 + eb - 1 with e0 = (lb % (kEll / eb)) eb.  Thread t takes local index t / eb of
// element e0 + t % eb, so the lanes of a warp hold one local index of consecutive elements: rows of one
// shape (equal trip counts through the row loops) whose entries lie side by side in the ELL slices.
struct ElemSlot {
  int i, t;   // the node and its slot, valid only if ok
  int el, l;  // the element's place in the block and the node's local index
  int g;      // the ELL group
  bool ok;
};
__device__ __forceinline__ ElemSlot element_slot(const Dev& D, int lb, int eb) {
  const int per_group = kEll / eb;
  const int g = lb / per_group;
  const int t = threadIdx.x;
  ElemSlot r;
  r.l = t / eb;
  r.el = t - r.l * eb;
  const int E = g * kEll + (lb - g * per_group) * eb + r.el;
  r.ok = r.l < D.n_loc && E < D.nel;
  r.i = E * D.n_loc + r.l;
  r.t = (g * D.n_loc + r.l) * kEll + (E & (kEll - 1));
  r.g = g;
  return r;
}

// Per node i of the block:
//  1. d_ij^H = max(d^min, d^ev) (Sec. 5, eq. (HighOrderViscosity); Sec. 5.1, eq. (ViscMin); Sec. 5.2),
//     the boundary d^{d,H} = max(c_k h_i^{p_k}, min(c_ev |N_i|, 1)) d^{d,L} (ghost node read as
//     collocated with x_i), and the high-order right-hand side
//       RHS^H_i = RHS^L_i - sum_j (d^H_ij - d^L_ij)(U_j - U_i) - sum_k (d^{d,H} - d^{d,L})(U^{d,k} - U_i);
//  2. the element solve of Sec. 5, eq. (HighScheme): dU^H_K = -tau M_K^{-1} RHS^H_K;
//  3. the relaxed bounds of Sec. 5.4, eq. (eq:local_bounds), from the one-hop aggregates of i and of
//     its stencil neighbours and node i's own boundary bar states;
//  4. A_ij = tau (d^H_ij - d^L_ij)(U_j - U_i) - m_ij (dU^H_j - dU^H_i) and
//     A_i^{d,k} = tau (d^{d,H} - d^{d,L})(U^{d,k} - U_i) (Sec. 5.3, eq. (HighLowOrderIdentity)), and the
//     pass-1 line search of Sec. 5.4, eq. (ConvexScheme), from U^L with P = A / (kappa_i m_i); the
//     searches that FP32 does not settle are queued for k_lsfix.
// With order HIGH the kernel stops after 2 and writes U_out = alpha U_base + (1 - alpha)(U + dU^H).
// The mixed path (MX) runs steps 1, 2 and the A_ij of step 4 in FP32 (the differences U_j - U_i in FP64
// first); the bounds and the line search stay FP64.
template <int DIM, bool MX, class Src>
__device__ __forceinline__ void high_sweep(const Src& src, int eb) {
  constexpr int M = DIM + 2;
  constexpr int kShared = kMaxBlock + kEll;        // room for one pad slot per element
  using R = std::conditional_t<MX, float, double>;  // arithmetic of steps 1, 2 and the A_ij of step 4
  __shared__ R sR[M][kShared];
  __shared__ int sE[kEll];  // 1 where some right-hand side of the element is not zero
  __shared__ R sdU[M][kShared];
  __shared__ Ctx sctx;
  int lb;
  const Ctx& c = src.get(&sctx, &lb);
  if (finished(c)) return;
  const Dev& D = c.D;
  const Scratch& S = c.S;
  const double* U = S.Us;
  const ElemSlot es = element_slot(D, lb, eb);
  const int i = es.t;
  const bool valid = es.ok;
  // the shared arrays space elements n_loc + 1 apart for even n_loc: the lanes of a warp read one node of
  // each of consecutive elements, and an even stride would put pairs of them in the same bank
  const int stride_sh = D.n_loc + !(D.n_loc & 1);
  const int t0 = es.el * stride_sh;  // the element's first slot in the shared arrays
  const int sh = t0 + es.l;
  const size_t n = D.ns;
  const double tau = stage_tau(c);
  for (int k = threadIdx.x; k < kEll; k += blockDim.x) sE[k] = 0;
  __syncthreads();
  const R tau_r = MX ? R(to_f32(tau)) : R(tau);
  double Ui[M];
  R rhs[M], dUi[M];
  double Ni = 0.0;
  const bool lim = D.order != GDG_ORDER_HIGH;  // the limiter's steps 3 and 4 follow the solve
  double lo = 0.0, hi = 0.0, sl = 0.0;         // two-hop aggregates of node i (step 3)
  bool quiet = true;                           // no viscous part of A in the row, and no boundary entry
  unsigned zeros = 0;                          // the stencil entries (of the row's first 32) without a viscous part
  if (valid) {
    load_state<DIM>(U, D.ns, i, Ui);
    Ni = abs_bits(S.N[i]);
#pragma unroll
    for (int q = 0; q < M; ++q) {
      if constexpr (MX)
        rhs[q] = to_f32(S.RHSL[(size_t)q * n + i]);
      else
        rhs[q] = S.RHSL[(size_t)q * n + i];
    }
    // min / max of non-negative values on the integer pipe; no thread of this body writes an input of the loop, so its
    // loads take the read-only path where that is defined (ld_stage) and may move ahead of the stores of A.  The same pass
    // over I(i) gathers the two-hop aggregates of the relaxed bounds (step 3).
    const int e1 = D.sten_end[i];
    if (lim) {
      lo = S.agg[i];
      hi = S.agg[n + i];
      sl = S.agg[2 * n + i];
    }
    // not unrolled: with its products on the integer pipe the loop body is large, and unrolled by 2 the
    // kernel stalled on instruction fetch (4.24 against 4.14 ms per launch at Q2 1024^2)
    unsigned bit = 1;  // of the entry in zeros; 0 from the row's 33rd entry on
#pragma unroll 1
    for (int e = D.rbeg[i]; e < e1; e += kEll, bit <<= 1) {  // I(i)
      const int j = __ldg(D.col + e);
      double Uj[M];
#pragma unroll
      for (int q = 0; q < M; ++q) Uj[q] = ld_stage<Src>(U + (size_t)q * n + j);
      if (lim) {
        lo = pmin(lo, ld_stage<Src>(S.agg + j));
        hi = pmax(hi, ld_stage<Src>(S.agg + n + j));
        sl = pmin(sl, ld_stage<Src>(S.agg + 2 * n + j));
      }
      bool same = true;
#pragma unroll
      for (int q = 0; q < M; ++q) same = same && same_bits(Ui[q], Uj[q]);
      if (same) {  // no viscous term; its zero is stored only where a row with other terms needs it
        zeros |= bit;
        if (bit == 0)
#pragma unroll
          for (int q = 0; q < M; ++q) S.A[(size_t)q * D.nnz + e] = 0.0;
        continue;
      }
      quiet = false;
      const double dl64 = ld_stage<Src>(S.dL + e), mu = __ldg(D.mu + e), Nj = abs_bits(ld_stage<Src>(S.N + j));
      if constexpr (MX) {
        // d^H - d^L from FP32 operands: every factor is symmetric in (i, j), so the same bits come out
        // of row j, and A_ji = -A_ij holds exactly
        const float dl = to_f32(dl64);
        const float dev = dl * fminf(D.c_ev_f * to_f32(pmax(Ni, Nj)), 1.f);
        const float dd = fmaxf(to_f32(mu) * dl, dev) - dl;
        const float td = tau_r * dd;
#pragma unroll
        for (int q = 0; q < M; ++q) {
          const float du = to_f32(Uj[q] - Ui[q]);
          rhs[q] = fmaf(-dd, du, rhs[q]);
          S.A[(size_t)q * D.nnz + e] = to_f64(td * du);  // viscous part of A_ij, completed below
        }
      } else {
        // products on the integer pipe (sf::mul, the same bits as the FP64 instruction)
        const double dl = dl64;
        const double dev = sf::mul(dl, pmin(sf::mul(D.c_ev, pmax(Ni, Nj)), 1.0));
        const double dd = pmax(sf::mul(mu, dl), dev) - dl;
        const double td = sf::mul(tau, dd);
#pragma unroll
        for (int q = 0; q < M; ++q) {
          const double du = Uj[q] - Ui[q];
          rhs[q] = fma(-dd, du, rhs[q]);
          S.A[(size_t)q * D.nnz + e] = sf::mul(td, du);  // viscous part of A_ij, completed below
        }
      }
    }
    for (int b = D.b_ptr[i]; b < D.b_ptr[i + 1]; ++b) {
      quiet = false;
      if (lim) {
        lo = pmin(lo, S.bbar[b]);
        hi = pmax(hi, S.bbar[b]);
        sl = pmin(sl, S.bbar[(size_t)D.nb + b]);
      }
      double UB[M];  // from the edge sweep
#pragma unroll
      for (int q = 0; q < M; ++q) UB[q] = S.UB[(size_t)q * D.nb + b];
      double dl = S.dB[b];
      double dd = (pmax(D.muB[i], pmin(D.c_ev * Ni, 1.0)) - 1.0) * dl;
#pragma unroll
      for (int q = 0; q < M; ++q) {
        if constexpr (MX)
          rhs[q] -= to_f32(dd * (UB[q] - Ui[q]));
        else
          rhs[q] -= dd * (UB[q] - Ui[q]);
        S.AB[(size_t)q * D.nb + b] = tau * dd * (UB[q] - Ui[q]);
      }
    }
    bool zero = true;
#pragma unroll
    for (int q = 0; q < M; ++q) {
      sR[q][sh] = rhs[q];
      if constexpr (MX)
        zero = zero && (__float_as_uint(rhs[q]) << 1) == 0u;
      else
        zero = zero && is_zero_bits(rhs[q]);
    }
    if (!zero) sE[es.el] = 1;
    if (lim) {  // relaxed local bounds, read back after the solve
      double rmin = 0.0, rmax = INFINITY, smin = 0.0;
      if (D.bounds_mode == 0) {
        rmin = D.rminus[i] * lo;
        rmax = D.rplus[i] * hi;
        smin = D.rminus[i] * sl;
      }
      S.bounds[i] = rmin;
      S.bounds[n + i] = rmax;
      S.bounds[2 * n + i] = smin;
    }
  }
  __syncthreads();
  // all right-hand sides of the element zero: so are dU^H and the mass terms of A
  const bool flat = sE[es.el] == 0;
  if (valid) {
    const int nl = D.n_loc;
    // row il of the element's M_K^{-1}, stored grouped like the entries: (E, a, b) at
    // ((E / kEll * n_loc + a) * n_loc + b) * kEll + E % kEll
    const double* Minv = D.MKinv + ((size_t)es.g * nl + es.l) * nl * kEll + (i & (kEll - 1));
    if (flat) {
#pragma unroll
      for (int q = 0; q < M; ++q) dUi[q] = R(0);
    } else {
      // FP64 multiply-adds, 36 of the kernel's 130 operations per node (Q2 quads).  In fixed point on the integer pipe
      // they are either less exact or no faster (fixdot.cuh).
      R acc[M];
#pragma unroll
      for (int q = 0; q < M; ++q) acc[q] = R(0);
      for (int l = 0; l < nl; ++l) {
        R w;
        if constexpr (MX)
          w = to_f32(__ldg(Minv + (size_t)l * kEll));
        else
          w = __ldg(Minv + (size_t)l * kEll);
#pragma unroll
        for (int q = 0; q < M; ++q) acc[q] += w * sR[q][t0 + l];
      }
#pragma unroll
      for (int q = 0; q < M; ++q) {
        if constexpr (MX)
          dUi[q] = -tau_r * acc[q];
        else
          dUi[q] = -tau * acc[q];
      }
    }
#pragma unroll
    for (int q = 0; q < M; ++q) sdU[q][sh] = dUi[q];
    if (D.order == GDG_ORDER_HIGH) {
#pragma unroll
      for (int q = 0; q < M; ++q) {
        double du;
        if constexpr (MX)
          du = to_f64(dUi[q]);
        else
          du = dUi[q];
        store_out(c, (size_t)q * D.n + es.i, rk_out(c, (size_t)q * D.n + es.i, U[(size_t)q * n + i] + du));
      }
    }
  }
  if (D.order == GDG_ORDER_HIGH) {
    if (valid) S.rem[i] = 3;
    return;
  }
  __syncthreads();
  const int nl = D.n_loc;
  const int se = valid ? D.sten_end[i] : 0, r0 = valid ? D.rbeg[i] : 0, r1 = valid ? D.rend[i] : 0;
  // Antidiffusive fluxes.  The mass term couples the nodes of one element, and A_ji = -A_ij: each pair is worked
  // out once, by the node that has at most half the element after it (cyclically), and stored at both
  // entries; half the FP64 operations of a loop in which every row does its own.
  // With dU^H = 0 the viscous part, which both rows have, is all there is; a row whose A is zero throughout is
  // marked instead of written: U^(1)_i = U^L_i whatever its factors, which are 1.
  quiet = quiet && flat;
  if (flat && !quiet) {
    unsigned bit = 1;
    for (int e = r0; e < r1; e += kEll, bit <<= 1)
      if (e >= se || (zeros & bit))
#pragma unroll
        for (int q = 0; q < M; ++q) S.A[(size_t)q * D.nnz + e] = 0.0;
  }
  unsigned bit = 1;
  for (int e = flat ? r1 : r0; e < r1; e += kEll, bit <<= 1) {
    const int j = D.col[e];
    const bool visc = e < se && !(zeros & bit);
    const int sj = j / kEll, gj = div_nl(D, sj);  // slice and group of j
    if (gj != es.g || ((j ^ i) & (kEll - 1)) != 0) {  // another element: no mass term
      if (!visc)
#pragma unroll
        for (int q = 0; q < M; ++q) S.A[(size_t)q * D.nnz + e] = 0.0;
      continue;
    }
    const int lj = sj - gj * nl;
    int after = lj - es.l;
    if (after < 0) after += nl;
    if (2 * after > nl || (2 * after == nl && lj < es.l)) continue;
    const int t = D.tr[e];
    if constexpr (MX) {
      const float mij = to_f32(D.mij[e]);
#pragma unroll
      for (int q = 0; q < M; ++q) {
        const float a = visc ? to_f32(S.A[(size_t)q * D.nnz + e]) : 0.f;
        const double v = to_f64(fmaf(-mij, sdU[q][t0 + lj] - dUi[q], a));
        S.A[(size_t)q * D.nnz + e] = v;
        S.A[(size_t)q * D.nnz + t] = sf::neg(v);
      }
    } else {
      const double mij = D.mij[e];
#pragma unroll
      for (int q = 0; q < M; ++q) {
        const double a = visc ? S.A[(size_t)q * D.nnz + e] : 0.0;
        const double v = fma(-mij, sdU[q][t0 + lj] - dUi[q], a);
        S.A[(size_t)q * D.nnz + e] = v;
        S.A[(size_t)q * D.nnz + t] = sf::neg(v);
      }
    }
  }
  __syncthreads();
  if (!valid) return;
  S.rem[i] = quiet ? 2 : 0;
  if (quiet) {
    for (int e = r0; e < r1; e += kEll) S.l1[e] = 1.0;
    return;
  }
  const double rmin = S.bounds[i], rmax = S.bounds[n + i], smin = S.bounds[2 * n + i];
  // pass-1 line search
  double UL[M];
#pragma unroll
  for (int q = 0; q < M; ++q) UL[q] = S.UL[(size_t)q * n + i];
  LsRow<DIM> ls;
  ls_row<DIM>(D, ls, UL, rmin, rmax, smin);
  const double ikm = D.inv_km[i];
  const float ikmf = d2f_fast(ikm);
  for (int e = r0; e < r1; e += kEll) {
    double A[M];
#pragma unroll
    for (int q = 0; q < M; ++q) A[q] = S.A[(size_t)q * D.nnz + e];
    // A = 0 (a uniform neighbourhood): the search's outcome is l = 1 exactly when the FP32 tests it
    // starts with pass, which here reduce to a density gap above and psi(0) > 0; then skip them
    unsigned long long abits = 0;
#pragma unroll
    for (int q = 0; q < M; ++q) abits |= (unsigned long long)__double_as_longlong(A[q]) << 1;
    if (abits == 0 && ls.dhi > 0.f && ls.psi0f > 0.f) {
      S.l1[e] = 1.0;
      continue;
    }
    double l;
    if (line_search_sure<DIM>(D, ls, A, ikm, ikmf, &l))
      S.l1[e] = l;
    else
      ls_defer(S, 0, e, i);
  }
  for (int b = D.b_ptr[i]; b < D.b_ptr[i + 1]; ++b) {
    double A[M];
#pragma unroll
    for (int q = 0; q < M; ++q) A[q] = S.AB[(size_t)q * D.nb + b];
    double l;
    if (line_search_sure<DIM>(D, ls, A, ikm, ikmf, &l))
      S.l1B[b] = l;
    else
      ls_defer(S, 0, -(b + 1), i);
  }
}

// The element sweep of each path as its own kernel with its own register budget.  Its loads, FP64 chains and 64-bit
// integer chains leave the issue slots half empty at 27 warps per SM, so a few spills are worth a fourth 288-thread
// block: in us per launch at 72, 56 and 48 registers 1,412, 1,268 and 1,211 (Q2 1024^2), 140, 109 and 114 (Q3 96^2), 239, 233
// and 252 (Q1 512^2), 390, 379 and 370 (Q1 48 x 40 x 44); the mixed path 302, 261 and 241 (Q2 384^2).
template <int DIM, class Src>
__global__ void __maxnreg__(56) k_high(Src src, int eb) {
  chain_begin();
  high_sweep<DIM, false, Src>(src, eb);
}
template <int DIM, class Src>
__global__ void __maxnreg__(72) k_high_few(Src src, int eb) {
  chain_begin();
  high_sweep<DIM, false, Src>(src, eb);
}
template <int DIM, class Src>
__global__ void __maxnreg__(48) k_high_mixed(Src src, int eb) {
  chain_begin();
  high_sweep<DIM, true, Src>(src, eb);
}

// eb: elements per block, a power of two <= kEll with eb * n_loc <= kMaxBlock (one element may exceed
// no block: n_loc <= kMaxLocal); n_loc is the one of the instance (a batch shares it).
template <int DIM, bool MX, class Src>
cudaError_t high_launch(const Src& src, long long blocks, int n_loc, int eb, cudaStream_t s) {
  if (blocks <= 0) return cudaSuccess;
  if (eb < 1 || eb > kEll || (eb & (eb - 1)) || n_loc < 1 || n_loc > kMaxLocal || eb * n_loc > kMaxBlock)
    return cudaErrorInvalidValue;
  const int threads = high_threads(n_loc, eb);
  if constexpr (MX) {
    return launch_chained(k_high_mixed<DIM, Src>, (unsigned)blocks, threads, s, src, eb);
  } else {
    if constexpr (std::is_same_v<Src, One>)
      if (few_threads(blocks, threads)) return launch_chained(k_high_few<DIM, Src>, (unsigned)blocks, threads, s, src, eb);
    return launch_chained(k_high<DIM, Src>, (unsigned)blocks, threads, s, src, eb);
  }
}

template <class Src>
cudaError_t high_dispatch(int dim, bool mx, const Src& src, long long blocks, int n_loc, int eb, cudaStream_t s) {
  switch (dim * 2 + (mx ? 1 : 0)) {
    case 2: return high_launch<1, false, Src>(src, blocks, n_loc, eb, s);
    case 3: return high_launch<1, true, Src>(src, blocks, n_loc, eb, s);
    case 4: return high_launch<2, false, Src>(src, blocks, n_loc, eb, s);
    case 5: return high_launch<2, true, Src>(src, blocks, n_loc, eb, s);
    case 6: return high_launch<3, false, Src>(src, blocks, n_loc, eb, s);
    case 7: return high_launch<3, true, Src>(src, blocks, n_loc, eb, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

#ifndef GDG_BODIES_ONLY  // (a file that includes this one for its kernel bodies defines it)
// eb: elements per block (all instances of a batch share n_loc, hence the block shape).
cudaError_t launch_high_file(int dim, const Ctx& c, long long blocks, int eb, cudaStream_t s) {
  return high_dispatch(dim, c.D.mixed != 0, One{c}, blocks, c.D.n_loc, eb, s);
}

cudaError_t launch_high_file_many(int dim, bool mixed, const Many& m, int n_loc, long long blocks, int eb,
                                  cudaStream_t s) {
  return high_dispatch(dim, mixed, m, blocks, n_loc, eb, s);
}

#endif  // GDG_BODIES_ONLY

}  // namespace gdg
