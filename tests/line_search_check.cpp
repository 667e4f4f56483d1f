// The deferred line search of csrc/gdg_internal.cuh compiled as host C++ (device_shim.h), against its root in long double.  The file
// named by argument 1 holds doubles: dim, gamma, count, then for every search U0, A, w, rho_min, rho_max, s_min.  An
// iterated search's error is measured in units of ls_tol + 2^-52 E / |psi'|, what its tolerance and psi's rounding leave open.
// Prints the root mean square and the ends of the errors; fails where the mean is above a half, an error above 3 (3 roundings of psi,
// whose terms are three), or an answer of the search infeasible by its own psi.
#include "device_shim.h"
#include "../paper_2402_04514_gb300/csrc/gdg_internal.cuh"

#include <stdio.h>
#include <vector>

using namespace gdg;

template <int DIM>
int run(double gamma, long n, FILE* f) {
  constexpr int M = DIM + 2;
  Dev D{};
  set_eos(D, gamma);
  D.ls_tol = 1e-14;
  D.ls_maxit = 50;
  std::vector<double> r(2 * M + 4);
  long double sq = 0, least = 0, most = 0;
  long count = 0, infeasible = 0;
  for (long k = 0; k < n; ++k) {
    if (fread(r.data(), sizeof(double), r.size(), f) != r.size()) return 2;
    const double *U0 = &r[0], *A = &r[M], w = r[2 * M], rmin = r[2 * M + 1], rmax = r[2 * M + 2], smin = r[2 * M + 3];
    const double got = line_search<DIM>(D, U0, A, w, rmin, rmax, smin);
    auto psi = [&](long double t) {
      const long double rho = U0[0] + t * w * A[0];
      long double m2 = 0;
      for (int q = 1; q <= DIM; ++q) m2 += (U0[q] + t * w * A[q]) * (U0[q] + t * w * A[q]);
      return U0[DIM + 1] + t * w * A[DIM + 1] - m2 / rho / 2 - smin * powl(rho, (long double)gamma);
    };
    const long double Pr = (long double)w * A[0];
    long double l = 1;
    if (U0[0] + Pr < rmin) l = (rmin - (long double)U0[0]) / Pr;
    if (U0[0] + Pr > rmax) l = (rmax - (long double)U0[0]) / Pr;
    l = std::min(std::max(l, 0.0L), 1.0L);
    if (psi(l) >= 0 || psi(0) < 0) continue;  // nothing to iterate
    long double a = 0, b = l;
    for (int it = 0; it < 80; ++it) ((psi((a + b) / 2) >= 0) ? a : b) = (a + b) / 2;
    double d;
    if (ls_psi_dpsi<DIM>(D, U0, A, got * w, smin, &d) < 0 && got > 0) ++infeasible;
    ls_psi_dpsi<DIM>(D, U0, A, (double)a * w, smin, &d);
    const long double e = (got - a) / (1e-14L + ldexpl(1, -52) * (U0[DIM + 1] + a * w * A[DIM + 1]) / fabsl((long double)d * w));
    ++count, sq += e * e, least = std::min(least, e), most = std::max(most, e);
  }
  printf("%ld searches: rms %.3Lf, %.2Lf to %.2Lf, %ld infeasible\n", count, sqrtl(sq / count), least, most, infeasible);
  return !(count > 0 && sqrtl(sq / count) <= 0.5L && least >= -3 && most <= 3 && infeasible == 0);
}

int main(int argc, char** argv) {
  FILE* f = argc > 1 ? fopen(argv[1], "rb") : nullptr;
  double h[3];
  if (!f || fread(h, sizeof(double), 3, f) != 3) return 2;
  const long n = (long)h[2];
  return h[0] == 1 ? run<1>(h[1], n, f) : h[0] == 2 ? run<2>(h[1], n, f) : run<3>(h[1], n, f);
}
