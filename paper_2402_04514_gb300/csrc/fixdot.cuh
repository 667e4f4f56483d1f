// Fixed-point dot products of binary64 vectors, on the host.
#pragma once
#include "fixfp64.cuh"

namespace sf {

// Dot products of binary64 vectors in fixed point: each vector as 56-bit integers below a common power of two, every
// integer in two 28-bit parts, so that a product is four 32 x 32 + 64-bit integer multiply-adds without rounding,
// packing or carries, in place of an FP64 multiply-add that holds its pipe 16 clocks per warp.  The three
// sums stay below 2^62 for up to 32 terms and are exact.  What is left out is what the operands lose: 2^-57 of
// their vector's largest power of two each, where the FP64 sum rounds every partial sum to 2^-54 of itself.
//
// No kernel takes this: an operand below an eighth of its vector's largest keeps fewer bits than its own 53, so that a sum whose
// large operands meet the other vector's small ones is further off than FP64's (27 terms, one of them large: 52.8 against
// 9.2 times 2^-53 of sum |a| |b| at most), and the element solve's FP64 loop, once the fluxes took its place on the FP64 pipe only
// once a pair, is no slower: in us per k_high launch 233 against 239 (Q1 512^2), 497 against 531 (32 Q1 meshes), 379 against
// 372 (Q1 48 x 40 x 44), 1,256 against 1,230 (Q2 1024^2), 107 against 99 (Q3 96^2).  A third part makes the sum as good as
// one rounding, at 283, 598, 397, 1,334 and 111 us.  It stands here, for the host alone, with its check.
//
// x in units of 2^(E - 1022 - 56), to nearest, for an exponent field E at least x's: below 2^56 in magnitude.
// A subnormal x counts as 0.
SF_FN int64_t fix56(double x, int E) {
  const int e = expo(x), d = E - e;
  const uint64_t s = e == 0 ? 0 : sig53(x) << 4;
  const uint64_t f = ((d < 63 ? s >> d : 0) + 1u) >> 1;
  return (hiw(x) >> 31) ? -(int64_t)f : (int64_t)f;
}
struct fixp {  // hi 2^28 + lo, 0 <= lo < 2^28
  int32_t hi, lo;
};
SF_FN fixp fix_parts(int64_t f) { return fixp{(int32_t)(f >> 28), (int32_t)((uint32_t)f & 0xfffffffu)}; }
SF_FN int64_t mad32(int32_t a, int32_t b, int64_t c) { return (int64_t)a * b + c; }
struct fixs {
  int64_t s1, s2, s3;  // the products of both high parts, of a high and a low part, of both low parts
};
SF_FN void fix_mad(fixp a, fixp b, fixs& s) {
  s.s1 = mad32(a.hi, b.hi, s.s1);
  s.s2 = mad32(a.hi, b.lo, mad32(a.lo, b.hi, s.s2));
  s.s3 = mad32(a.lo, b.lo, s.s3);
}
// s1 2^56 + s2 2^28 + s3 in units of 2^(Ea - 1022 - 56) 2^(Eb - 1022 - 56), rounded to binary64
SF_FN double fix_dbl(const fixs& s, int Ea, int Eb) {
  const int64_t s2 = s.s2 + (s.s3 >> 28);
  int64_t t = s.s1 + (s2 >> 28);
  uint64_t f = (uint64_t)s2 << 36;  // the 28 bits below t, at the top of the word
  const bool ng = t < 0;
  if (ng) {
    f = 0 - f;
    t = f ? ~t : -t;
  }
  int e = Ea + Eb - 2100 + 63;
  uint64_t h = (uint64_t)t;
  if (h == 0) h = f >> 36, f = 0, e -= 28;
  if (h == 0) return 0.0;
  const uint32_t hh = (uint32_t)(h >> 32);
  const int z = hh ? (int)clz32(hh) : 32 + (int)clz32((uint32_t)h);
  h = z == 0 ? h : (h << z) | (f >> (64 - z));
  const double r = uf_dbl(uf{h, e - z});
  return ng ? neg(r) : r;
}

}  // namespace sf
