// Deferred line searches (csrc/gdg_internal.cuh as host C++, device_shim.h) along directions in which psi is flat to its rounding:
// U0 + t A moves along an isentrope, psi(0) is 1e-17 to 1e-15 of the energy and psi(1) below 0 by its curvature alone.  Any
// point whose psi comes out non-negative is as good as another then, but a search must not give up on the far part of the
// segment: against the bracketed iteration (ls_maxit = 7 chooses it) no more searches may end at 0, and the mean of the
// factors may be 5% smaller at most.
#include "device_shim.h"
#include "../paper_2402_04514_gb300/csrc/gdg_internal.cuh"

#include <stdio.h>

using namespace gdg;

static unsigned long long state = 88172645463325252ull;
static double uniform() {  // xorshift64
  state ^= state << 13, state ^= state >> 7, state ^= state << 17;
  return (double)(state >> 11) * 0x1p-53;
}

int main() {
  Dev D{};
  set_eos(D, 1.4);
  D.ls_tol = 1e-14;
  double sum[2] = {0, 0};
  long zero[2] = {0, 0}, count = 0;
  for (long k = 0; k < 400000; ++k) {
    const double rho = 0.5 + uniform(), v = uniform() - 0.5, eps = (0.5 + uniform()) / 0.4;
    const double U0[3] = {rho, rho * v, eps + 0.5 * rho * v * v};
    const double dr = pow(10.0, -9 + 4 * uniform()) * (uniform() < 0.5 ? 1 : -1);
    const double A[3] = {dr, v * dr, 1.4 * eps / rho * dr + 0.5 * v * v * dr};
    const double smin = eps / pow(rho, 1.4) * (1 - pow(10.0, -17 + 2 * uniform()));
    double l[2], d;
    for (int q = 0; q < 2; ++q) {
      D.ls_maxit = q ? 7 : 50;
      l[q] = line_search<1>(D, U0, A, 1.0, 0.0, 10.0, smin);
    }
    if (l[0] == 1.0 || ls_psi_dpsi<1>(D, U0, A, 0.0, smin, &d) < 0) continue;
    ++count;
    for (int q = 0; q < 2; ++q) sum[q] += l[q], zero[q] += l[q] == 0;
  }
  printf("%ld searches: mean %.4f, %ld at 0; bracketed %.4f, %ld at 0\n", count, sum[0] / count, zero[0], sum[1] / count, zero[1]);
  return !(count > 100000 && zero[0] <= zero[1] && sum[0] >= 0.95 * sum[1]);
}
