// The fixed-point dot product of csrc/fixfp64.cuh, compiled as host C++, against long double and against the FP64 sum it stands
// for.  Standard input: n, then the n x n matrix as hexadecimal floats; arguments: vectors, seed.  The vectors spread over 0 to 40
// binary orders, some with zeros.  Prints the root mean square and the largest error of both, relative to |row| |vector| (in
// the largest entries), and fails where the fixed-point ones are the larger or above their bound.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <random>
#include <vector>

#include "../paper_2402_04514_gb300/csrc/fixfp64.cuh"

int main(int argc, char** argv) {
  int n;
  if (argc < 3 || scanf("%d", &n) != 1 || n < 1 || n > 32) return 2;
  std::vector<double> M(n * n), r(n);
  for (double& v : M)
    if (scanf("%la", &v) != 1) return 2;
  std::mt19937_64 g(atol(argv[2]));
  std::uniform_real_distribution<double> uni(-1.0, 1.0);
  long double sq[2] = {0, 0}, mx[2] = {0, 0};
  const long N = atol(argv[1]);
  for (long k = 0; k < N; ++k) {
    const int spread = (int)(k % 41), off = (int)(g() % 600) - 300;
    int Er = 0;
    double rmax = 0;
    for (double& v : r) {
      v = k % 7 == 6 && g() % 2 ? 0.0 : ldexp(uni(g), off - (spread ? (int)(g() % spread) : 0));
      Er = std::max(Er, sf::expo(v)), rmax = std::max(rmax, fabs(v));
    }
    for (int a = 0; a < n; ++a) {
      const double* w = &M[a * n];
      int Ew = 0;
      double wmax = 0, plain = 0;
      for (int l = 0; l < n; ++l) Ew = std::max(Ew, sf::expo(w[l])), wmax = std::max(wmax, fabs(w[l]));
      sf::fixs s{0, 0, 0};
      long double want = 0;
      for (int l = 0; l < n; ++l) {
        sf::fix_mad(sf::fix_parts(sf::fix56(w[l], Ew)), sf::fix_parts(sf::fix56(r[l], Er)), s);
        plain = fma(w[l], r[l], plain);
        want += (long double)w[l] * r[l];
      }
      const double got[2] = {sf::fix_dbl(s, Ew, Er), plain};
      for (int q = 0; q < 2; ++q) {
        const long double e = rmax > 0 ? fabsl(got[q] - want) / ((long double)wmax * rmax) : fabsl((long double)got[q]);
        sq[q] += e * e, mx[q] = std::max(mx[q], e);
      }
    }
  }
  const long double u = ldexpl(1, -53), cnt = (long double)N * n;
  printf("n %d: fixed rms %.3Lf max %.3Lf, FP64 rms %.3Lf max %.3Lf (2^-53)\n", n, sqrtl(sq[0] / cnt) / u, mx[0] / u,
         sqrtl(sq[1] / cnt) / u, mx[1] / u);
  // per term: half a unit of 2^-56 from each operand, whose power of two is below twice its maximum: 2^-56 of it; then one
  // rounding, to half an ulp, of a sum of at most n products
  return sq[0] > sq[1] || mx[0] > n * 2 * ldexpl(1, -56) + n * u;
}
