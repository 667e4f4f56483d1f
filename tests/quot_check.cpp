// The integer quotient of csrc/fixfp64.cuh compiled as host C++ against the processor's division, bit for bit: argument 1 the
// number of operand pairs, 2 the seed.  Random significands, both close to 1, equal, near 2, one a power of two, quotients within a
// few units of a rounding boundary, exact quotients; exponents near each other and far apart; both signs.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <random>

#include "../paper_2402_04514_gb300/csrc/fixfp64.cuh"

int main(int argc, char** argv) {
  const long n = argc > 1 ? atol(argv[1]) : 100000;
  std::mt19937_64 g(argc > 2 ? atol(argv[2]) : 0);
  const uint64_t F = 0xfffffffffffffULL;
  long checked = 0;
  for (long k = 0; k < n; ++k) {
    uint64_t fa = g() & F, fb = g() & F;
    switch (k % 8) {
      case 1: fa &= 0xff, fb &= 0xff; break;
      case 2: fa = fb + g() % 5 - 2; break;
      case 3: fa |= F - 0xff, fb |= F - 0xff; break;
      case 4: (k & 8 ? fa : fb) = 0; break;
      default: break;
    }
    const int ea = k % 3 ? 1000 + (int)(g() % 40) : 1 + (int)(g() % 2046), eb = k % 3 ? 1000 + (int)(g() % 40) : 1 + (int)(g() % 2046);
    const uint64_t sg = g() & 0x8000000000000000ULL, sh = g() & 0x8000000000000000ULL;
    double a = sf::dbl(sg | ((uint64_t)ea << 52) | (fa & F));
    const double b = sf::dbl(sh | ((uint64_t)eb << 52) | (fb & F));
    if (k % 8 == 5) a = b * (1.0 + (double)(g() % 1000) * 0x1p-52);                        // close to a representable quotient
    if (k % 8 == 6) a = fma(b, 1.0 + ((double)(g() >> 12) + 0.5) * 0x1p-52, 0.0);          // close to half way
    if (k % 8 == 7) a = (double)(float)b * (double)(float)(1.0 + (double)(g() >> 44) * 0x1p-20);  // often exact
    if (!sf::quot_ok(a, b)) continue;
    ++checked;
    const double got = sf::quot(a, b), want = a / b;
    if (!(got == want)) return printf("%a / %a: %a, want %a\n", a, b, got, want), 1;
  }
  printf("%ld of %ld\n", checked, n);
  return checked < n / 2;
}
