// Reciprocals, square roots, inverse q-th roots and integer powers of binary64 numbers on the integer pipe.
//
// The GB300's FP64 pipe retires 2 thread-operations per clock per SM and answers after 64 clocks; a 64 x 64-bit
// integer product takes a quarter of that pipe time and 35 to 40 clocks.  These routines take the FP32
// approximation of the special-function unit as a 24-bit integer, form the exact residual of the defining
// equation (1 - x y, 1 - s y, 1 - x y^q) in 64-bit integers, where the leading bits cancel and need not be kept,
// and add the first terms of the binomial series.  What they compute is good to about 2^-59 of the value
// before the one rounding to binary64 at the end, so every result is within 0.52 ulp of the exact one; the
// Newton steps in FP64 that they replace were good to 1 or 2 ulp.
//
// Products that follow (powers) stay unpacked, as a 64-bit significand and an exponent: without rounding,
// packing and special cases a product is a third of the instructions of sf::mul and carries 11 more bits.
// Per launch at Q2 1024^2: k_edge 3.09 -> 2.18 ms, k_prim 0.81 -> 0.45, k_high 3.81 -> 3.67.
//
// The integer path covers positive normal operands (for the reciprocal, normal ones of either sign); the
// callers take the FP64 operation for everything else.  The header compiles as host C++ too, where the
// integer code is checked against long double.
#pragma once
#include <math.h>

#include "softfp64.cuh"

namespace sf {

SF_FN uint64_t mulhi64(uint64_t a, uint64_t b) {
#if defined(__CUDA_ARCH__)
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
SF_FN uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
SF_FN uint32_t fbits(float x) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(x);
#else
  uint32_t u;
  memcpy(&u, &x, sizeof u);
  return u;
#endif
}
SF_FN float flt(uint32_t u) {
#if defined(__CUDA_ARCH__)
  return __uint_as_float(u);
#else
  float x;
  memcpy(&x, &u, sizeof x);
  return x;
#endif
}

// The special-function unit's approximations (relative error below 2^-22 for the arguments they get here).  On the host
// rounded double values stand for them, passed through SF_HOST_APPROX, by which a check can move them within the
// instructions' documented errors.
#ifndef SF_HOST_APPROX
#define SF_HOST_APPROX(y) (y)
#endif
SF_FN float mufu_rcp(float x) {
#if defined(__CUDA_ARCH__)
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return (float)SF_HOST_APPROX(1.0 / x);
#endif
}
SF_FN float mufu_rsqrt(float x) {
#if defined(__CUDA_ARCH__)
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return (float)SF_HOST_APPROX(1.0 / sqrt((double)x));
#endif
}
SF_FN float mufu_lg2(float x) {
#if defined(__CUDA_ARCH__)
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return (float)SF_HOST_APPROX(log2((double)x));
#endif
}
SF_FN float mufu_ex2(float x) {
#if defined(__CUDA_ARCH__)
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return (float)SF_HOST_APPROX(exp2((double)x));
#endif
}

// A positive number m 2^(e - 63), 2^63 <= m < 2^64.
struct uf {
  uint64_t m;
  int e;
};

// The exponent field of x, and whether x is a positive normal number.
SF_FN int expo(double x) { return (int)((hiw(x) >> 20) & 0x7ffu); }
SF_FN bool pos_normal(double x) { return hiw(x) - 0x00100000u < 0x7fe00000u; }
// the 53-bit significand
SF_FN uint64_t sig53(double x) { return (((uint64_t)((hiw(x) & 0xfffffu) | 0x100000u)) << 32) | low(x); }
// the significand in [1, 2) as FP32, truncated
SF_FN float sigf(double x) { return flt(0x3f800000u | ((hiw(x) & 0xfffffu) << 3) | (low(x) >> 29)); }

SF_FN uf uf_of(double x) { return uf{sig53(x) << 11, expo(x) - 1023}; }  // positive normal x
SF_FN uf uf_mul(uf a, uf b) {
  uint64_t h = mulhi64(a.m, b.m);  // in [2^62, 2^64)
  const int top = (int)(h >> 63);
  return uf{h << (1 - top), a.e + b.e + top};
}
// Rounded to nearest (ties, which only exact products reach, upwards).  Outside the normal range: by two
// scalings in FP64, out of line.
#if defined(__CUDA_ARCH__)
static __device__ __noinline__ __attribute__((const)) double uf_far(uint64_t m, int e) { return ldexp((double)m, e - 63); }
#else
static inline double uf_far(uint64_t m, int e) { return ldexp((double)m, e - 63); }
#endif
SF_FN double uf_dbl(uf a) {
  const uint64_t s = (a.m >> 11) + ((a.m >> 10) & 1u);  // 2^53 after a carry: the addition moves it on
  if (__builtin_expect((unsigned)(a.e + 1022) >= 2044u, 0)) return uf_far(a.m, a.e);
  return dbl(((uint64_t)(uint32_t)(a.e + 1022) << 52) + s);
}
// x^k, k >= 1, by binary powering
SF_FN uf uf_pow(uf x, int k) {
  while (!(k & 1)) {
    x = uf_mul(x, x);
    k >>= 1;
  }
  uf r = x;
  while (k >>= 1) {
    x = uf_mul(x, x);
    if (k & 1) r = uf_mul(r, x);
  }
  return r;
}

// The 24-bit significand of an approximation y of a number in [1/2, 1], in units of 2^-24.  y itself may lie an ulp or two below
// 1/2 (the reciprocal of a number just below 2, the inverse square root of one just below 4), where its exponent
// would give a negative shift: 1/2 is then the better approximation.
SF_FN uint32_t sig_half(float y) {
  const uint32_t u = fbits(y), b = u < 0x3f000000u ? 0x3f000000u : u;
  return ((b & 0x7fffffu) | 0x800000u) << ((b >> 23) - 126u);
}

// 1 / m for the significand m of x in [1, 2), in units of 2^-63: at most 2^63, which m = 1 gives.  With Y the
// 24-bit approximation and e = 1 - m Y (below 2^-21), 1 / m = Y (1 + e + e^2 + ...): the residual
// -M Y modulo 2^64 (M Y is near 2^76, a multiple of 2^64), then Y e and Y e^2; Y e^3 is below 2^-63.
SF_FN uint64_t rcp_sig(double x) {
  const uint32_t mh = (hiw(x) & 0xfffffu) | 0x100000u, ml = low(x);
  const uint32_t Y = sig_half(mufu_rcp(sigf(x)));
  const uint64_t MY = wide(ml, Y) + ((uint64_t)(mh * Y) << 32);
  const int64_t r = -(int64_t)MY;  // e in units of 2^-76
  const int32_t rh = (int32_t)(r >> 32);
  const uint32_t rl = (uint32_t)r;
  // Y e in units of 2^-68
  const int64_t c1 = (int64_t)rh * (int64_t)(int32_t)Y + (int64_t)(wide(rl, Y) >> 32);
  // Y e^2: e = rh 2^-44, e^2 = rh^2 2^-88
  const uint32_t e2 = (uint32_t)((uint64_t)((int64_t)rh * rh) >> 20);  // units of 2^-68
  const uint32_t c2 = (uint32_t)(wide(e2, Y) >> 24);                   // units of 2^-68
  return ((uint64_t)Y << 39) + (uint64_t)((c1 + (int64_t)c2) >> 5);
}
// 1 / x for a normal x whose reciprocal is normal (rcp_ok)
SF_FN bool rcp_ok(double x) { return (unsigned)(expo(x) - 1) < 2043u; }
SF_FN double rcp(double x) {
  const uint64_t T = rcp_sig(x) + 512u;
  const uint64_t r = ((uint64_t)(uint32_t)(2044 - expo(x)) << 52) + (T >> 10);
  return dbl(r | ((uint64_t)(hiw(x) & 0x80000000u) << 32));
}
SF_FN uf uf_rcp(double x) {  // positive normal x
  const uint64_t T = rcp_sig(x);
  const int one = (int)(T >> 63);
  return uf{T << (1 - one), 1022 - expo(x) + one};
}

// a / b for normal a and b with a quotient well inside the normal range (quot_ok), correctly rounded: a 53-bit quotient from
// the reciprocal, at most one off, and the exact remainder, whose size says whether it is and how to round (a quotient
// of two 53-bit numbers is never half way between two others).
SF_FN bool quot_ok(double a, double b) {
  const int ea = expo(a), eb = expo(b);
  return (unsigned)(ea - 1) < 2046u && (unsigned)(eb - 1) < 2046u && (unsigned)(ea - eb + 1000) < 2000u;
}
SF_FN double quot(double a, double b) {
  const uint64_t A = sig53(a), B = sig53(b);
  const int below = A < B;                                              // the quotient of the significands is below 1
  uint64_t q = mulhi64(A << 11, rcp_sig(b)) >> (10 - below);            // in units of 2^-52, below 1 of 2^-53
  int64_t r = (int64_t)((A << (52 + below)) - q * B);                   // modulo 2^64; between -B and 2 B
  const int less = r < 0, more = r >= (int64_t)B;
  q += (uint64_t)more - (uint64_t)less;
  r += less ? (int64_t)B : more ? -(int64_t)B : 0;
  q += 2 * r > (int64_t)B;  // 2^53 after a carry: the addition below moves it on
  const uint64_t e = (uint64_t)(uint32_t)(expo(a) - expo(b) + 1022 - below);
  return dbl(((e << 52) + q) | ((uint64_t)((hiw(a) ^ hiw(b)) & 0x80000000u) << 32));
}

// sqrt(x) for a positive normal x.  X in [1, 4) is x with an even power of two taken out, Y the 24-bit
// approximation of X^{-1/2}, s = X Y and e = 1 - s Y (below 2^-20): sqrt(X) = s (1 - e)^{-1/2} =
// s (1 + e/2 + 3/8 e^2 + ...), the next term below 2^-61.
SF_FN double sqrt_pos(double x) {
  const int ex = expo(x), odd = (ex & 1) ^ 1;  // 1023 is odd: an even field is an odd power of two
  const uint64_t X = sig53(x) << odd;          // units of 2^-52, below 2^54
  const uint32_t Y = sig_half(mufu_rsqrt(flt(fbits(sigf(x)) + ((uint32_t)odd << 23))));
  const uint32_t xh = (uint32_t)(X >> 32), xl = (uint32_t)X;
  // s = X Y in units of 2^-60: (X Y) >> 16, X Y below 2^78
  const uint64_t p0 = wide(xl, Y), p1 = wide(xh, Y) + (p0 >> 32);
  const uint64_t s = (p1 << 16) | ((uint32_t)p0 >> 16);
  const uint32_t sh = (uint32_t)(s >> 32), sl = (uint32_t)s;
  const int64_t r = -(int64_t)(wide(sl, Y) + ((uint64_t)(sh * Y) << 32));  // e in units of 2^-84
  const int32_t rh = (int32_t)(r >> 32);                                   // units of 2^-52
  const uint32_t rl = (uint32_t)r;
  // s e / 2 in units of 2^-60: (s r) 2^-144 / 2 = (s r) >> 85 units, from the upper products
  const int64_t hi = (int64_t)rh * (int64_t)(int32_t)sh + (int64_t)(wide(sh, rl) >> 32) +
                     (((int64_t)rh * (int64_t)(sl >> 1)) >> 31);  // (s r) >> 64; sh is below 2^29
  const int32_t eh = (int32_t)(r >> 40);                            // units of 2^-44, below 2^24
  const uint32_t e2 = (uint32_t)((uint64_t)((int64_t)eh * eh) >> 22);  // units of 2^-66
  const uint64_t c2 = (wide(e2, (uint32_t)(s >> 37)) * 3u) >> 32;     // 3/8 s e^2: 2^-89 -> 2^-60 is >> 29, and / 8
  const uint64_t T = s + (uint64_t)(hi >> 21) + c2 + 128u;
  return dbl(((uint64_t)(uint32_t)(((ex + 1023 - (odd ? 1 : 0)) >> 1) - 1) << 52) + (T >> 8));
}

// Constants of the inverse q-th root, 1 <= q <= 16.
struct rootc {
  int q;
  float iqf;       // 1 / q
  uint32_t qdiv;   // ceil(2^20 / q): floor(u / q) = (u qdiv) >> 20 for u < 2^20 / q
  uint32_t c2;     // (q + 1) / (2 q^2) in units of 2^-24
  uint64_t iq;     // 1 / q in units of 2^-64 (2^64 - 1 for q = 1)
};
SF_FN rootc root_const(int q) {
  rootc r;
  r.q = q;
  r.iqf = 1.0f / (float)q;
  r.qdiv = ((1u << 20) + (uint32_t)q - 1u) / (uint32_t)q;
  r.c2 = (uint32_t)(((((uint64_t)q + 1u) << 24) + (uint64_t)q * q) / (2u * (uint64_t)q * (uint64_t)q));
  r.iq = q == 1 ? ~(uint64_t)0 : (uint64_t)((~(uint64_t)0) / (uint64_t)q);
  return r;
}

// x^{-1/q} for a positive normal x.  x = X 2^a with X in [1, 2), -a = q b + c with 0 <= c < q: the approximation
// is 2^b y, y = exp2((c - log2 X) / q), its argument in (-1, 1), so that it is as good far from 1 as near it.  y is
// taken as a 24-bit significand Y in [1, 2) and an exponent; X Y^q is 2^k (1 - t) for a known k with
// |t| below 2^-17, and x^{-1/q} = y (1 - t)^{-1/q} = y (1 + t / q + (q + 1) / (2 q^2) t^2 + ...), the next term below
// 2^-59 (its factor is at most 0.1 for q >= 3; for q = 1, 2 t is below 2^-20).
SF_FN uf uf_rootinv(double x, const rootc& c) {
  const int a = expo(x) - 1023;
  const uint32_t u = (uint32_t)(1024 * c.q - a);
  const int b = (int)((u * c.qdiv) >> 20);  // floor(-a / q) + 1024
  const int rem = (int)u - c.q * b;
  const float yf = mufu_ex2(((float)rem - mufu_lg2(sigf(x))) * c.iqf);
  const uint32_t yb = fbits(yf);
  const uint32_t Y = (yb & 0x7fffffu) | 0x800000u;
  const int ye = (int)(yb >> 23) - 127;  // y = Y 2^-23 2^ye
  // X Y^q as an unpacked product, 2^k (1 - t)
  const uf p = uf_mul(uf_pow(uf{(uint64_t)Y << 40, 0}, c.q), uf{sig53(x) << 11, 0});
  // t in units of 2^-63: the product is just below 2^k (p.m near 2^64, p.e = k - 1) or just above (near 2^63)
  const bool above = !(p.m >> 62 & 1u);
  const int64_t t = above ? -(int64_t)(p.m & 0x7fffffffffffffffULL) : (int64_t)((0 - p.m) >> 1);
  const bool neg = t < 0;
  const uint64_t at = (uint64_t)(neg ? -t : t);  // below 2^46
  // delta = t / q + c2 t^2 in units of 2^-60
  const uint64_t d1 = mulhi64(at << 16, c.iq) >> 19;
  const uint32_t ts = (uint32_t)(at >> 24);                                // units of 2^-39, below 2^22
  const uint64_t d2 = (uint64_t)((uint32_t)(wide(ts, ts) >> 18)) * c.c2 >> 24;  // t^2 in units of 2^-60, times c2
  const int64_t d = (neg ? -(int64_t)d1 : (int64_t)d1) + (int64_t)d2;
  const uint64_t T = ((uint64_t)Y << 39) + (uint64_t)((d * (int64_t)(int32_t)Y) >> 21);  // units of 2^-62
  const int lz = (int)clz32((uint32_t)(T >> 32));  // 0, 1 or 2
  return uf{T << lz, b - 1024 + ye + 1 - lz};
}

}  // namespace sf

#if !defined(__CUDACC__)
#include "fixdot.cuh"
#endif
