// Low-order sweep: per-node primitives, the time-step reduction (Sec. 3.3, eq. (MaxCFLdt)) and the
// first stage sweep (low-order update, entropy-viscosity indicator, one-hop bound aggregates).
// Every kernel takes its context from a source (One: a single instance, Many: a batch; gdg_internal.cuh).
#include <type_traits>

#include "gdg_internal.cuh"

namespace gdg {

namespace {

constexpr int kThreads = kRowMaxThreads;  // launch bound; the schedule launches 128, 256 or 512

// Per-node primitives (Sec. 2.2): 1/rho, p, 1/p, a = sqrt(gamma p / rho), p^{-e}, the entropy function
// f(s) = exp(s / (gamma + 1)) of the entropy-viscosity indicator and s~ = rho^{-gamma} eps (Sec. 5.4).
// Flags a state outside the admissible set of eq. (AddSet).  Being the first kernel of every stage, it
// also empties the stage's deferred line-search queues.  The mixed path (MX) keeps 1/rho and p in FP64
// (the fluxes use them) and computes the rest in FP32.  With c.Ucopy set (the first stage of a step whose
// state comes from host memory, read here over the host link) it also stores the state it read there, for
// the later sweeps of the stage; when the instance's clock has finished, the step is a no-op and it also
// writes that state to c.Uhost, the step's host output, where the last stage's writers would have.
template <int DIM, bool MX, class Src>
__device__ __forceinline__ void prim_body(const Src& src) {
  __shared__ Ctx sctx;
  int lb;
  const Ctx& c = src.get(&sctx, &lb);
  const bool done = finished(c);
  if (done && !c.Ucopy) return;
  const Dev& D = c.D;
  const Scratch& S = c.S;
  const int slot = lb * blockDim.x + threadIdx.x;
  if (slot == 0 && !done) {
    S.lsq_n[0] = 0u;
    S.lsq_n[1] = 0u;
  }
  // by slots, so that the nine or more arrays written here are; over the host link the reads decide
  const Node nd = row_node(D, slot, c.Ucopy == nullptr);
  const int i = nd.i, t = nd.t;
  if (i < 0) return;
  double Ui[DIM + 2];
  load_state<DIM>(c.U, D.n, i, Ui);
  if (c.Ucopy) {
#pragma unroll
    for (int q = 0; q < DIM + 2; ++q) c.Ucopy[(size_t)q * D.n + i] = Ui[q];
    if (done) {
      if (c.Uhost)
#pragma unroll
        for (int q = 0; q < DIM + 2; ++q) c.Uhost[(size_t)q * D.n + i] = Ui[q];
      return;
    }
  }
  const size_t n = D.ns;
#pragma unroll
  for (int q = 0; q < DIM + 2; ++q) S.Us[q * n + t] = Ui[q];
  double irho = rcp64(Ui[0]);
  // products on the integer pipe (sf::mul, the same bits as the FP64 instruction) where no sum follows
  double m2 = sf::mul(Ui[1], Ui[1]);
#pragma unroll
  for (int k = 1; k < DIM; ++k) m2 = fma(Ui[1 + k], Ui[1 + k], m2);
  double eps = fma(-sf::mul_pow2(m2, -1), irho, Ui[DIM + 1]);
  if (!(Ui[0] > 0.0) || !(eps > 0.0)) atomicOr(S.flags, (unsigned)GDG_FLAG_INADMISSIBLE);
  double p = sf::mul(D.gm1, eps);
  double* P = S.prim;
  if constexpr (MX) {
    const PrimF f = prim_mx(D, Ui[0], p);
    float st = powf(to_f32(Ui[0]), -D.gamma_f) * to_f32(eps);
    double st64 = to_f64(st);
    if (!finite_f32(st)) {  // rho^{-gamma} beyond the FP32 range
      double ir;
      st64 = rho_neg_gamma(D, Ui[0], &ir) * eps;
      st = to_f32(st64);
    }
    P[PR_IRHO * n + t] = irho;
    P[PR_P * n + t] = p;
    P[PR_IP * n + t] = to_f64(f.ip);
    P[PR_A * n + t] = to_f64(f.a);
    P[PR_PME * n + t] = to_f64(f.pme);
    P[PR_F * n + t] = to_f64(powf(2.f * D.gm1h_f * st, D.inv_gp1_f));
    P[PR_ST * n + t] = st64;
    return;
  }
  double ir;
  double st = sf::mul(rho_neg_gamma(D, Ui[0], &ir), eps);
  P[PR_IRHO * n + t] = irho;
  P[PR_P * n + t] = p;
  P[PR_IP * n + t] = rcp64(p);
  P[PR_A * n + t] = sqrt64(sf::mul(sf::mul(D.gamma, p), irho));
  P[PR_PME * n + t] = D.ie_root > 0 ? rootinv(p, D.root_ie) : pow_hw(p, -D.e_exp);
  // f = (gm1 s~)^{1/(gamma+1)} = x^{q/(p+q)} = x (x^{-1/(p+q)})^p for gamma = p/q
  double x = sf::mul(D.gm1, st);
  P[PR_F * n + t] = (D.gq > 0 && D.gp + D.gq <= 16 && sf::pos_normal(x))
                        ? sf::uf_dbl(sf::uf_mul(sf::uf_of(x), sf::uf_pow(sf::uf_rootinv(x, D.root_gpq.c), D.gp)))
                        : pow_hw(x, D.inv_gp1);
  P[PR_ST * n + t] = st;
}

template <int DIM, bool MX, class Src>
__global__ void __launch_bounds__(kThreads) k_prim(Src src) {
  chain_begin();
  prim_body<DIM, MX, Src>(src);
}

// Boundary entry b of a stage: the unit normal, the interior and the boundary state, their m.n, v.n and pressures, and
// d_i^{d,k} = |c_i^{d,k}| lambda_max^+(U_i, U^{d,k}, n_i^k) (Sec. 4.2, eq. (eq:dij_low_order_modified); interior state on
// the left).
template <int DIM>
struct Side {
  double n[DIM], Ui[DIM + 2], UB[DIM + 2], mnL, mnR, uL, uR, pL, pB, d;
};
template <int DIM, bool MX>
__device__ __forceinline__ void boundary_side(const Ctx& c, int b, Side<DIM>& o) {
  const Dev& D = c.D;
  const double* P = c.S.prim;
  const size_t n = D.ns, nb = D.nb;
  const int i = D.bnode[b];
  load_state<DIM>(c.S.Us, D.ns, i, o.Ui);
  const double irL = P[PR_IRHO * n + i];
  o.pL = P[PR_P * n + i];
#pragma unroll
  for (int k = 0; k < DIM; ++k) o.n[k] = D.bn[(size_t)k * nb + b];
  boundary_state<DIM>(D, b, o.Ui, c.bdata, o.n, o.UB);
  const double irB = rcp64(o.UB[0]);
  o.pB = sf::mul(D.gm1, fma(-sf::mul_pow2(dot<DIM>(o.UB + 1, o.UB + 1), -1), irB, o.UB[DIM + 1]));
  o.mnL = dot<DIM>(o.Ui + 1, o.n);
  o.mnR = dot<DIM>(o.UB + 1, o.n);
  o.uL = sf::mul(o.mnL, irL);
  o.uR = sf::mul(o.mnR, irB);
  double ipB, aB, pmeB;
  prim_of<MX>(D, o.UB[0], irB, o.pB, &ipB, &aB, &pmeB);
  o.d = sf::mul(D.bnorm[b], lambda_pair<MX>(D, o.uL, o.pL, irL, P[PR_IP * n + i], P[PR_A * n + i], P[PR_PME * n + i], o.uR,
                                            o.pB, irB, ipB, aB, pmeB));
}

// Block minimum of val, then one 64-bit atomicMin per block on the bit pattern (positive doubles order
// like uint64).  Every thread of the block calls it.
__device__ __forceinline__ void block_min_to(double val, unsigned long long* dst) {
  __shared__ double red[kThreads / 32];
  for (int off = 16; off > 0; off >>= 1) val = fmin(val, __shfl_xor_sync(0xffffffffu, val, off));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = val;
  __syncthreads();
  if (threadIdx.x < 32) {
    val = threadIdx.x < blockDim.x / 32 ? red[threadIdx.x] : INFINITY;
    for (int off = 16; off > 0; off >>= 1) val = fmin(val, __shfl_xor_sync(0xffffffffu, val, off));
    if (threadIdx.x == 0 && val < INFINITY) atomicMin(dst, (unsigned long long)__double_as_longlong(val));
  }
}

// d_ij^L of every stencil edge and d_i^{d,k} of every boundary entry (gdg_max_dt, before any stage), one thread
// per boundary entry and then one per undirected edge as in the edge sweep below, stored for the row sums of k_tau
// in arrays that the next stage overwrites before it reads them.  By edges each bound is worked out once
// where a loop over rows does it twice, and no boundary row holds up its warp: 23 -> 8 us per call with
// the row sums at Q2 33 x 47.
template <int DIM, bool MX, class Src>
__device__ __forceinline__ void maxdt_body(const Src& src) {
  __shared__ Ctx sctx;
  int lb;
  const Ctx& c = src.get(&sctx, &lb);
  if (finished(c)) return;
  const Dev& D = c.D;
  const Scratch& S = c.S;
  const double* P = S.prim;
  const size_t n = D.ns, nnz = D.nnz;
  const unsigned slot = lb * blockDim.x + threadIdx.x, nbs = boundary_slots(D.nb);
  if (slot < nbs) {
    if (slot >= (unsigned)D.nb) return;
    Side<DIM> side;
    boundary_side<DIM, MX>(c, (int)slot, side);
    S.bbar[slot] = side.d;
    return;
  }
  const unsigned k = slot - nbs;
  if (k >= (unsigned)D.ne) return;
  const int e = D.edge_e[k], i = D.edge_i[k], j = D.col[e];
  double nv[DIM], mi[DIM], mj[DIM];
#pragma unroll
  for (int q = 0; q < DIM; ++q) {
    nv[q] = D.cn[q * nnz + e];
    mi[q] = S.Us[(1 + q) * n + i];
    mj[q] = S.Us[(1 + q) * n + j];
  }
  const double ir_i = P[PR_IRHO * n + i], ir_j = P[PR_IRHO * n + j];
  const double uL = sf::mul(dot<DIM>(mi, nv), ir_i), uR = sf::mul(dot<DIM>(mj, nv), ir_j);
  const double d = sf::mul(D.cnorm[e], lambda_pair<MX>(D, uL, P[PR_P * n + i], ir_i, P[PR_IP * n + i], P[PR_A * n + i],
                                                       P[PR_PME * n + i], uR, P[PR_P * n + j], ir_j, P[PR_IP * n + j],
                                                       P[PR_A * n + j], P[PR_PME * n + j]));
  S.psi[e] = d;  // (l1, where barR lies, stays the last stage's)
  S.psi[D.tr[e]] = d;
}

template <int DIM, bool MX, class Src>
__global__ void __launch_bounds__(kThreads) k_maxdt(Src src) {
  chain_begin();
  maxdt_body<DIM, MX, Src>(src);
}

// Sums over the rows of d_ij^L plus the boundary viscosities, i.e. -d_ii of eq. (eq:dij_low_order_supplement), then
// min over nodes of m_i / (2 |d_ii|): inside a fused step (with a clock) from what the edge sweep of its first
// stage stored, into the clock; for gdg_max_dt from what k_maxdt stored.  Capped at 48 registers: the row
// sum is latency-bound and wants many warps.
template <int DIM, bool MX, class Src>
__device__ __forceinline__ void tau_body(const Src& src, int sliced) {
  __shared__ Ctx sctx;
  int lb;
  const Ctx& c = src.get(&sctx, &lb);
  if (finished(c)) return;
  const Dev& D = c.D;
  const Scratch& S = c.S;
  const Node nd = row_node(D, lb * blockDim.x + threadIdx.x, sliced);
  const int i = nd.t;
  const double* dL = c.clk ? S.dL : S.psi;
  const double* dB = c.clk ? S.dB : S.bbar;
  double val = INFINITY;
  if (nd.i >= 0) {
    double dsum = 0.0;
    const int e0 = D.rbeg[i], e1 = D.sten_end[i];
#pragma unroll 4
    for (int e = e0; e < e1; e += kEll) dsum += ld_stage<Src>(dL + e);  // loads issued ahead of the in-order sum
    for (int b = D.b_ptr[i], b1 = D.b_ptr[i + 1]; b < b1; ++b) dsum += dB[b];
    if (dsum > 0.0) val = sf::mul(sf::mul_pow2(D.mi[i], -1), rcp64(dsum));
  }
  block_min_to(val, c.clk ? &c.clk->tau_bits : S.tau_bits);
}

template <int DIM, bool MX, class Src>
__global__ void __maxnreg__(48) k_tau(Src src, int sliced) {
  chain_begin();
  tau_body<DIM, MX, Src>(src, sliced);
}

// s~ of a state in the mixed path, from rho, |m|^2 / 2 and E: eps in FP64 (E - |m|^2 / (2 rho) cancels at high Mach
// numbers) with 1/rho from one Newton step on the FP32 reciprocal; rho^{-gamma} in FP32.
__device__ __forceinline__ double entropy_mx(const Dev& D, double rho, double hm2, double E) {
  const float rf = to_f32(rho);
  const double y = to_f64(1.f / rf);
  double ir = __dmul_rn(y, fma(-rho, y, 2.0));
  const float rg = powf(rf, -D.gamma_f);
  if (finite_f32(rg)) return to_f64(__fmul_rn(rg, to_f32(fma(-hm2, ir, E))));
  const double rg64 = rho_neg_gamma(D, rho, &ir);
  return rg64 * fma(-hm2, ir, E);
}

// What a stage needs of boundary entry b, one thread per entry (the first threads of the edge sweep, so that
// the sweeps over rows read it instead of working it out inside their rows: the powers, roots and
// divisions of an entry are a chain of FP64 operations that held up its row's whole warp, in every sweep
// again): the boundary state (Sec. 4.1), d_i^{d,k} = |c_i^{d,k}| lambda_max^+(U_i, U^{d,k}, n_i^k)
// (Sec. 4.2, eq. (eq:dij_low_order_modified); interior state on the left), both fluxes times c_i^{d,k},
// and rho and s~ of the boundary bar state (eq. (BoundaryBarState)).  At Q2 301 x 259 with open sides, in us per
// launch: k_low 326 -> 213, k_tau 138 -> 34, k_high 414 -> 322, k_edge 241 -> 245.  A function of its own, so
// that its registers are not the edges': inlined, the edges spill 136 bytes in place of 44.
template <int DIM, bool MX>
__device__ __noinline__ void boundary_entry(const Ctx& c, int b) {
  constexpr int M = DIM + 2;
  const Dev& D = c.D;
  const Scratch& S = c.S;
  const size_t nb = D.nb;
  Side<DIM> o;
  boundary_side<DIM, MX>(c, b, o);
  const double cnm = D.bnorm[b], d = o.d;
  const double *Ui = o.Ui, *UB = o.UB;
  S.dB[b] = d;
  double fi[M], fB[M], Ub[M];
  flux_n<DIM>(Ui, o.n, o.mnL, o.uL, o.pL, fi);
  flux_n<DIM>(UB, o.n, o.mnR, o.uR, o.pB, fB);
  const double t = sf::mul(sf::mul_pow2(cnm, -1), rcp64(d));
#pragma unroll
  for (int q = 0; q < M; ++q) {
    S.UB[q * nb + b] = UB[q];
    S.gB[q * nb + b] = sf::mul(cnm, fB[q]);
    S.gI[q * nb + b] = sf::mul(cnm, fi[q]);
    Ub[q] = fma(-t, fB[q] - fi[q], sf::mul_pow2(Ui[q] + UB[q], -1));
  }
  double irb;
  const double rg = rho_neg_gamma(D, Ub[0], &irb);
  S.bbar[b] = Ub[0];
  S.bbar[nb + b] = sf::mul(rg, fma(-sf::mul_pow2(dot<DIM>(Ub + 1, Ub + 1), -1), irb, Ub[DIM + 1]));
}

// Edge sweep, one thread per undirected stencil edge {i, j} (i < j): the quantities of a pair that are
// symmetric in i and j are computed once and written to both entries (i, j) and (j, i):
//  - d_ij^L = d_ji^L = |c_ij| lambda_max^+(U_i, U_j, n_ij) (Sec. 3.1, eq. (eq:dij_low_order); the bound
//    is symmetric under (U_i, U_j, n) -> (U_j, U_i, -n), which is also what makes d^L symmetric);
//  - the bar state Ubar_ij = Ubar_ji (eq. (UsualBarState)), of which only rho is kept, and the least s~ of it
//    and both nodes (for the local bounds of eq. (eq:local_bounds));
//  - the flux difference G_ij = (f(U_j) - f(U_i)) c_ij = G_ji, whose row sums sweep A takes in place of those of
//    f(U_j) c_ij (they differ by f(U_i) sum_j c_ij, which Lemma LemPart gives in boundary terms): one symmetric
//    array where f(U_j) c_ij and f(U_i) c_ji were two, so that a row reads only its own entries.  With the
//    indicator's entry term computed here too, sweep A's loop has 14 FP64 operations per entry in place of 19
//    and 44 bytes less to read (2.49 -> 1.89 ms per launch at Q2 1024^2);
//  - the indicator's term (m_j . c_ij)(f_j - f_i) of Sec. 5.2 for both rows.
// The first threads take the boundary entries.
// The mixed path (MX) takes lambda from lambda_pair<true> and the entropy power of the bar state in FP32;
// the fluxes, G and the bar state itself stay FP64.
template <int DIM, bool MX, class Src>
__device__ __forceinline__ void edge_body(const Src& src) {
  constexpr int M = DIM + 2;
  __shared__ Ctx sctx;
  int lb;
  const Ctx& c = src.get(&sctx, &lb);
  if (finished(c)) return;
  const Dev& D = c.D;
  const Scratch& S = c.S;
  const unsigned slot = lb * blockDim.x + threadIdx.x, nbs = boundary_slots(D.nb);
  if (slot < nbs) {
    if (slot < (unsigned)D.nb) boundary_entry<DIM, MX>(c, (int)slot);
    return;
  }
  const unsigned k = slot - nbs;
  if (k >= (unsigned)D.ne) return;
  const size_t n = D.ns, nnz = D.nnz;
  const int e = D.edge_e[k], i = D.edge_i[k];
  const int j = D.col[e], t = D.tr[e];
  const double* P = S.prim;
  double Ui[M], Uj[M], nv[DIM];
  load_state<DIM>(S.Us, D.ns, i, Ui);
  load_state<DIM>(S.Us, D.ns, j, Uj);
  const double cnm = D.cnorm[e];
  // products on the integer pipe (sf::mul, the same bits as the FP64 instruction) where no sum follows
#pragma unroll
  for (int q = 0; q < DIM; ++q) nv[q] = D.cn[(size_t)q * nnz + e];
  double mnL = sf::mul(Ui[1], nv[0]), mnR = sf::mul(Uj[1], nv[0]);
#pragma unroll
  for (int q = 1; q < DIM; ++q) {
    mnL = fma(Ui[1 + q], nv[q], mnL);
    mnR = fma(Uj[1 + q], nv[q], mnR);
  }
  const double p_i = P[PR_P * n + i], p_j = P[PR_P * n + j];
  const double ir_i = P[PR_IRHO * n + i], ir_j = P[PR_IRHO * n + j];
  const double uL = sf::mul(mnL, ir_i), uR = sf::mul(mnR, ir_j);
  const double lam = lambda_pair<MX>(D, uL, p_i, ir_i, P[PR_IP * n + i], P[PR_A * n + i], P[PR_PME * n + i], uR, p_j,
                                     ir_j, P[PR_IP * n + j], P[PR_A * n + j], P[PR_PME * n + j]);
  const double d = sf::mul(cnm, lam);
  S.dL[e] = d;
  S.dL[t] = d;
  // Equal states, as in every region that no wave has reached: the differences are zero and the bar state is the
  // state itself, so the sweeps over rows, which see it from the states, take nothing but d_ij from the entry.
  // In ms per launch at Q2 1024^2, where the waves have crossed a few percent of the mesh: k_edge 2.22 -> 0.95, k_low
  // 1.89 -> 0.97, k_high 3.20 -> 1.51, k_limit2 0.96 -> 0.51.  Where no two states agree the tests cost 2% of a
  // step (Q1 512^2 vortex: k_high 237 -> 246 us, k_edge 196 -> 199, k_low 187 -> 183).
  bool same = true;
#pragma unroll
  for (int q = 0; q < M; ++q) same = same && same_bits(Ui[q], Uj[q]);
  if (same) return;
  // f(U) c_ij with c_ij = |c_ij| n_ij, from m.c = |c| m.n and v.c = |c| v.n
  double cv[DIM], gi[M], gj[M];
#pragma unroll
  for (int q = 0; q < DIM; ++q) cv[q] = sf::mul(cnm, nv[q]);
  flux_n<DIM>(Ui, cv, sf::mul(cnm, mnL), sf::mul(cnm, uL), p_i, gi);
  flux_n<DIM>(Uj, cv, sf::mul(cnm, mnR), sf::mul(cnm, uR), p_j, gj);
  // W = 2 Ubar = U_i + U_j - (f(U_j) - f(U_i)) c_ij / d_ij, halved where it is used
  const double r = MX ? to_f64(1.f / to_f32(d)) : rcp64(d);
  double W[M];
#pragma unroll
  for (int q = 0; q < M; ++q) {
    const double df = gj[q] - gi[q];
    S.G[q * nnz + e] = df;
    S.G[q * nnz + t] = df;
    W[q] = fma(-r, df, Ui[q] + Uj[q]);
  }
  if constexpr (MX) {
    S.psi[e] = gj[0];
    S.psi[t] = -gi[0];
  } else {
    const double fd = P[PR_F * n + j] - P[PR_F * n + i];
    S.psi[e] = sf::mul(gj[0], fd);
    S.psi[t] = sf::mul(gi[0], fd);  // (-gi)(f_i - f_j)
  }
  double Ub[M];
  Ub[0] = sf::mul_pow2(W[0], -1);
  Ub[DIM + 1] = sf::mul_pow2(W[DIM + 1], -1);
  double mw2 = sf::mul(W[1], W[1]);  // |2 m(Ubar)|^2; 0.125 mw2 = |m(Ubar)|^2 / 2
#pragma unroll
  for (int q = 1; q < DIM; ++q) mw2 = fma(W[1 + q], W[1 + q], mw2);
  const double hm2 = sf::mul_pow2(mw2, -3);
  double stb;
  if constexpr (MX) {
    stb = entropy_mx(D, Ub[0], hm2, Ub[DIM + 1]);
  } else {
    double irb;
    const double rgb = rho_neg_gamma(D, Ub[0], &irb);  // sets irb = 1 / rho(Ubar) before its use below
    stb = sf::mul(rgb, fma(-hm2, irb, Ub[DIM + 1]));
  }
  S.barR[e] = Ub[0];
  S.barR[t] = Ub[0];
  stb = pmin(stb, pmin(P[PR_ST * n + i], P[PR_ST * n + j]));
  S.barS[e] = stb;
  S.barS[t] = stb;
}

// Two 512-thread blocks per SM (64 registers, a few bytes of spills): the integer-pipe products of the
// sweep want resident warps to hide their latency.
template <int DIM, bool MX, class Src>
__global__ void __launch_bounds__(kThreads, 2) k_edge(const __grid_constant__ Src src) {
  chain_begin();
  edge_body<DIM, MX, Src>(src);
}

// Sweep A, one thread per row i, after the edge sweep:
//  - the row sums of d_ij^L and f(U_j) c_ij and the boundary terms, all from the edge sweep;
//  - the low-order update of Sec. 4.2, eq. (cijdijschememodified), and the CFL check (CFLcond);
//  - the entropy-viscosity indicator N_i = R_i / D_i (Sec. 5.2);
//  - the one-hop aggregates of the local bounds (Sec. 5.4, eq. (eq:local_bounds)): min/max of rho_j,
//    rho(Ubar_jk), rho_k and min of s~ over node j's stencil, with the bar states of
//    eq. (UsualBarState).
// With order LOW (or no limiter pass) it also writes U_out = alpha U_base + (1 - alpha) U^L.
// The mixed path (MX) computes the indicator in FP32 (its sums from FP64 flux differences); the low-order
// update stays FP64.
template <int DIM, bool MX, class Src>
__device__ __forceinline__ void low_body(const Src& src, int sliced, int write_out) {
  constexpr int M = DIM + 2;
  __shared__ Ctx sctx;
  int lb;
  const Ctx& c = src.get(&sctx, &lb);
  if (finished(c)) return;
  const Dev& D = c.D;
  const Scratch& S = c.S;
  const double* U = S.Us;
  const Node nd = row_node(D, lb * blockDim.x + threadIdx.x, sliced && !(write_out && c.Uhost));
  if (nd.i < 0) return;
  const int i = nd.t;
  const double tau = stage_tau(c);
  size_t n = D.ns;
  const double* P = S.prim;
  double Ui[M];
  load_state<DIM>(U, D.ns, i, Ui);
  const double irho_i = P[PR_IRHO * n + i], ip_i = P[PR_IP * n + i], f_i = P[PR_F * n + i],
               st_i = P[PR_ST * n + i];
  using Acc = std::conditional_t<MX, float, double>;  // arithmetic of the indicator's sums
  // RHS^L = sum_j f(U_j) c_ij - sum_j d_ij (U_j - U_i) + boundary terms, accumulated as its two sums
  // (sg, sdu); the indicator's sum is sg
  double sg[M], sdu[M];
  Acc Fsum[M];  // (mixed only)
#pragma unroll
  for (int q = 0; q < M; ++q) {
    sg[q] = sdu[q] = 0.0;
    Fsum[q] = Acc(0);
  }
  Acc psum = Acc(0);
  double dsum = 0.0;
  double lo = Ui[0], hi = Ui[0], sl = st_i;
  const size_t nnz = D.nnz;
  const int e1 = D.sten_end[i];
  bool active = D.b_ptr[i + 1] > D.b_ptr[i];  // some sum of the row has a term that is not zero
  bool equal = false;                         // some neighbour has the row's state
  for (int e = D.rbeg[i]; e < e1; e += kEll) {  // I(i)
    const int j = D.col[e];
    const double d = S.dL[e];
    dsum += d;
    double Uj[M];
    load_state<DIM>(U, D.ns, j, Uj);
    bool same = true;
#pragma unroll
    for (int q = 0; q < M; ++q) same = same && same_bits(Ui[q], Uj[q]);
    if (same) {  // equal states: the edge sweep's terms are zeros, and the extrema stay
      equal = true;
      continue;
    }
    active = true;
#pragma unroll
    for (int q = 0; q < M; ++q) {
      const double ge = S.G[q * nnz + e];
      sg[q] += ge;
      sdu[q] = fma(d, Uj[q] - Ui[q], sdu[q]);
      if constexpr (MX) Fsum[q] += to_f32(ge);  // the mixed path sums the FP64 differences in FP32
    }
    if constexpr (MX)
      psum += to_f32(S.psi[e]) * (to_f32(P[PR_F * n + j]) - to_f32(f_i));
    else
      psum += S.psi[e];
    lo = pmin(lo, pmin(Uj[0], S.barR[e]));
    hi = pmax(hi, pmax(Uj[0], S.barR[e]));
    sl = pmin(sl, S.barS[e]);
  }
  if constexpr (MX) {
    // the bar state of equal states is the state, but its s~ is rounded otherwise in FP32 than k_prim's
    if (equal) sl = pmin(sl, entropy_mx(D, Ui[0], sf::mul_pow2(dot<DIM>(Ui + 1, Ui + 1), -1), Ui[DIM + 1]));
  }
  // sg is now the sum of (f(U_j) - f(U_i)) c_ij; with the boundary terms, Fsum = sg - f(U_i) sum_k c_i^{d,k} =
  // sum_j f(U_j) c_ij and the right-hand side takes Fsum + sum_k f(U^{d,k}) c_i^{d,k}.  On a stencil that
  // holds one state every term is zero, or cancels with its partner, exactly.
  double sgB[M];
#pragma unroll
  for (int q = 0; q < M; ++q) sgB[q] = 0.0;
  for (int b = D.b_ptr[i], b1 = D.b_ptr[i + 1]; b < b1; ++b) {
    const size_t nb = D.nb;
    const double d = S.dB[b];
    dsum += d;
#pragma unroll
    for (int q = 0; q < M; ++q) {
      const double gi = S.gI[q * nb + b];
      sgB[q] += S.gB[q * nb + b];
      sg[q] -= gi;
      sdu[q] = fma(d, S.UB[q * nb + b] - Ui[q], sdu[q]);
      if constexpr (MX) Fsum[q] -= to_f32(gi);
    }
  }
  const double inv_mi = D.inv_mi[i];
  if (sf::mul(sf::mul(sf::mul_pow2(tau, 1), dsum), inv_mi) > 1.0 + 1e-12) atomicOr(S.flags, (unsigned)GDG_FLAG_CFL);
  double rhs[M], UL[M];
#pragma unroll
  for (int q = 0; q < M; ++q) rhs[q] = 0.0, UL[q] = Ui[q];
  if (active) {
    const double tm = -sf::mul(tau, inv_mi);
#pragma unroll
    for (int q = 0; q < M; ++q) {
      rhs[q] = (sg[q] + sgB[q]) - sdu[q];
      UL[q] = fma(tm, rhs[q], Ui[q]);
    }
  }
  if (write_out) {
#pragma unroll
    for (int q = 0; q < M; ++q) store_out(c, (size_t)q * D.n + nd.i, rk_out(c, (size_t)q * D.n + nd.i, UL[q]));
    return;
  }
#pragma unroll
  for (int q = 0; q < M; ++q) {
    S.UL[(size_t)q * n + i] = UL[q];
    S.RHSL[(size_t)q * n + i] = rhs[q];
  }
  S.agg[i] = lo;
  S.agg[n + i] = hi;
  S.agg[2 * n + i] = sl;
  if (!active) {
    S.N[i] = 0.0;
    return;
  }
  // entropy-viscosity indicator: Fsum_k = sum_j (f_k(U_j) - f_k(U_i)) c_ij - f_k(U_i) sum_k c_i^{d,k}, which
  // equals sum_j f_k(U_j) c_ij by the partition of unity (Lemma LemPart) and vanishes exactly on a
  // stencil holding one state; grad Phi_i = rho_i f'(s_i) grad_U s(U_i), f' = f / (gamma + 1),
  // grad_U s = grad_U p / p - (gamma / rho) e_rho, grad_U p = (gamma - 1)[|v|^2 / 2, -v, 1]
  if constexpr (MX) {
    const float irf = to_f32(irho_i), ipf = to_f32(ip_i), gm1 = 2.f * D.gm1h_f;
    const float pref = to_f32(f_i) * D.inv_gp1_f * to_f32(Ui[0]);
    float v[DIM], v2 = 0.f;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      v[k] = to_f32(Ui[1 + k]) * irf;
      v2 += v[k] * v[k];
    }
    float grad[M];
    grad[0] = pref * fmaf(D.gm1h_f * v2, ipf, -(D.gamma_f * irf));
#pragma unroll
    for (int k = 0; k < DIM; ++k) grad[1 + k] = pref * (-gm1 * v[k] * ipf);
    grad[DIM + 1] = pref * (gm1 * ipf);
    float R = psum, Dn = fabsf(psum);
#pragma unroll
    for (int q = 0; q < M; ++q) {
      R -= grad[q] * Fsum[q];
      Dn += fabsf(grad[q]) * fabsf(Fsum[q]);
    }
    S.N[i] = Dn > 0.f ? to_f64(R / Dn) : 0.0;
  } else {
    // rho f / (gamma + 1) from rho itself and 1/p from k_prim, so that no division is needed here
    const double pref = sf::mul(sf::mul(f_i, D.inv_gp1), Ui[0]);
    const double ip = ip_i;
    double vk[DIM];
#pragma unroll
    for (int k = 0; k < DIM; ++k) vk[k] = sf::mul(Ui[1 + k], irho_i);
    double v2 = sf::mul(vk[0], vk[0]);
#pragma unroll
    for (int k = 1; k < DIM; ++k) v2 = fma(vk[k], vk[k], v2);
    double grad[M];
    grad[0] = sf::mul(pref, fma(sf::mul(sf::mul(D.gm1, 0.5), v2), ip, -sf::mul(D.gamma, irho_i)));
#pragma unroll
    for (int k = 0; k < DIM; ++k) grad[1 + k] = sf::mul(pref, sf::mul(sf::mul(-D.gm1, vk[k]), ip));
    grad[DIM + 1] = sf::mul(pref, sf::mul(D.gm1, ip));
    double R = psum, Dn = fabs(psum);
#pragma unroll
    for (int q = 0; q < M; ++q) {
      R = fma(-grad[q], sg[q], R);
      Dn = fma(fabs(grad[q]), fabs(sg[q]), Dn);
    }
    S.N[i] = Dn > 0.0 ? sf::mul(R, rcp64(Dn)) : 0.0;
  }
}

// Four 256-thread blocks per SM (three in 3D): the row sums wait for loads and for the FP64 pipe.  In us per launch at
// 78 to 106 registers, at 64 (80) and at 48 (64): 845, 728 and 745 (Q2 1024^2), 181, 175 and 178 (Q1 512^2), 218, 206 and
// 208 (Q1 48 x 40 x 44); mixed 209, 154 and 166 (Q2 384^2).
template <int DIM, bool MX, class Src>
__global__ void __maxnreg__(DIM == 3 ? 80 : 64) k_low(Src src, int sliced, int write_out) {
  chain_begin();
  low_body<DIM, MX, Src>(src, sliced, write_out);
}
template <int DIM, bool MX, class Src>
__global__ void __launch_bounds__(kThreads) k_low_few(Src src, int sliced, int write_out) {
  chain_begin();
  low_body<DIM, MX, Src>(src, sliced, write_out);
}

template <int DIM, bool MX, class Src>
cudaError_t low_launch(int kern, const Src& src, long long blocks, int threads, int sliced, int arg, cudaStream_t s) {
  if (blocks <= 0) return cudaSuccess;
  if (threads < 32 || threads > kThreads || threads % 32) return cudaErrorInvalidValue;
  const unsigned g = (unsigned)blocks;
  switch (kern) {
    case KN_PRIM: return launch_chained(k_prim<DIM, MX, Src>, g, threads, s, src);
    case KN_MAXDT: return launch_chained(k_maxdt<DIM, MX, Src>, g, threads, s, src);
    case KN_TAU: return launch_chained(k_tau<DIM, MX, Src>, g, threads, s, src, sliced);
    case KN_EDGE: return launch_chained(k_edge<DIM, MX, Src>, g, threads, s, src);
    case KN_LOW:
      if constexpr (std::is_same_v<Src, One>)
        if (few_threads(blocks, threads)) return launch_chained(k_low_few<DIM, MX, Src>, g, threads, s, src, sliced, arg);
      return launch_chained(k_low<DIM, MX, Src>, g, threads, s, src, sliced, arg);
    default: return cudaErrorInvalidValue;
  }
}

template <class Src>
cudaError_t low_dispatch(int kern, int dim, bool mx, const Src& src, long long blocks, int threads, int sliced,
                         int arg, cudaStream_t s) {
  switch (dim * 2 + (mx ? 1 : 0)) {
    case 2: return low_launch<1, false, Src>(kern, src, blocks, threads, sliced, arg, s);
    case 3: return low_launch<1, true, Src>(kern, src, blocks, threads, sliced, arg, s);
    case 4: return low_launch<2, false, Src>(kern, src, blocks, threads, sliced, arg, s);
    case 5: return low_launch<2, true, Src>(kern, src, blocks, threads, sliced, arg, s);
    case 6: return low_launch<3, false, Src>(kern, src, blocks, threads, sliced, arg, s);
    case 7: return low_launch<3, true, Src>(kern, src, blocks, threads, sliced, arg, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

#ifndef GDG_BODIES_ONLY  // (a file that includes this one for its kernel bodies defines it)
// Launchers of this file's kernels, dispatched on the dimension and the precision (called by
// launch_kernel*).
cudaError_t launch_low_file(int kern, int dim, const Ctx& c, long long blocks, int threads, int sliced, int arg,
                            cudaStream_t s) {
  return low_dispatch(kern, dim, c.D.mixed != 0, One{c}, blocks, threads, sliced, arg, s);
}

cudaError_t launch_low_file_many(int kern, int dim, bool mixed, const Many& m, long long blocks, int threads,
                                 int sliced, int arg, cudaStream_t s) {
  return low_dispatch(kern, dim, mixed, m, blocks, threads, sliced, arg, s);
}

#endif  // GDG_BODIES_ONLY

}  // namespace gdg
