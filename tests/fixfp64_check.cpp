// Checks csrc/fixfp64.cuh compiled as host C++ against long double: argument 1 the number of operands, 2 the seed.  Operands:
// any exponent, exponents near 1, significands at both ends of [1, 2), and exact powers of two.  Prints the largest
// errors; exit status 1 where one exceeds its bound.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <random>

#include "../paper_2402_04514_gb300/csrc/fixfp64.cuh"

static long double ulps(double got, long double want) {
  const double w = fabs((double)want);
  return fabsl((long double)got - want) / (long double)(nextafter(w, INFINITY) - w);
}
static long double value(sf::uf a) { return ldexpl((long double)a.m, a.e - 63); }

int main(int argc, char** argv) {
  const long n = argc > 1 ? atol(argv[1]) : 100000;
  std::mt19937_64 g(argc > 2 ? atol(argv[2]) : 0);
  long double rcp = 0, sq = 0, root = 0, urcp = 0, uroot = 0, umul = 0, upow = 0;
  for (long k = 0; k < n; ++k) {
    uint64_t m = g() & 0xfffffffffffffULL;
    int ex = 1021 + (int)(g() % 5);
    switch (k % 5) {
      case 0: ex = 1 + (int)(g() % 2043); break;
      case 1: m &= 0xff; break;
      case 2: m |= 0xfffffffffff00ULL; break;
      case 3: m = 0, ex = 1 + (int)(g() % 2043); break;
      default: break;
    }
    const double x = sf::dbl(((uint64_t)ex << 52) | m);
    const long double X = x;
    if (sf::rcp_ok(x)) {
      rcp = fmaxl(rcp, ulps(sf::rcp(x), 1.0L / X));
      rcp = fmaxl(rcp, ulps(-sf::rcp(-x), 1.0L / X));
    }
    urcp = fmaxl(urcp, fabsl(value(sf::uf_rcp(x)) * X - 1.0L));
    sq = fmaxl(sq, ulps(sf::sqrt_pos(x), sqrtl(X)));
    const int q = 1 + (int)(k % 16);
    const sf::uf y = sf::uf_rootinv(x, sf::root_const(q));
    // powl rounds 1 / q, which far from 1 costs up to 2^-55 of the value: one Newton step on x r^q = 1 repairs it
    long double ref = powl(X, -1.0L / q), prod = X;
    for (int f = 0; f < q; ++f) prod *= ref;
    ref += ref * (1.0L - prod) / q;
    if (!(y.m >> 63)) return printf("not normalised: %a q %d\n", x, q), 1;
    uroot = fmaxl(uroot, fabsl(value(y) / ref - 1.0L));
    root = fmaxl(root, ulps(sf::uf_dbl(y), ref));
    const double z = sf::dbl(((uint64_t)(1000 + g() % 40) << 52) | (g() & 0xfffffffffffffULL));
    const double w = sf::dbl(((uint64_t)(1000 + g() % 40) << 52) | (g() & 0xfffffffffffffULL));
    umul = fmaxl(umul, fabsl(value(sf::uf_mul(sf::uf_of(z), sf::uf_of(w))) / ((long double)z * w) - 1.0L));
    const int p = 1 + (int)(g() % 12);
    upow = fmaxl(upow, fabsl(value(sf::uf_pow(sf::uf_of(z), p)) / powl(z, p) - 1.0L));
  }
  printf("rcp %.4Lf sqrt %.4Lf root %.4Lf ulp; unpacked rcp 2^%.2f root 2^%.2f mul 2^%.2f pow 2^%.2f\n", rcp, sq, root,
         log2((double)urcp), log2((double)uroot), log2((double)umul), log2((double)upow));
  // one rounding (0.5 ulp) plus what the fixed-point terms leave: 2^-57 of the value is 1/16 ulp at most
  return rcp > 0.5625L || sq > 0.5625L || root > 0.5625L || urcp > ldexpl(1, -60) || uroot > ldexpl(1, -57) ||
         umul > ldexpl(1, -61) || upow > 12 * ldexpl(1, -61);
}
