// Host check of csrc/fixsum.h: sums of seven values with the stencil's signs
// against long-double sums.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "fixsum.h"

using namespace kfbim;

static double stencil(const double* u) {   // u1 + .. + u6 - 6 u0
  int E = kFixMin;
  for (int k = 0; k < 7; ++k) E = std::max(E, fix_exp(cvt_bits64(u[k])));
  int64_t s = -6 * fix_of(cvt_bits64(u[0]), E);
  for (int k = 1; k < 7; ++k) s += fix_of(cvt_bits64(u[k]), E);
  return fix_value(s, E);
}

int main() {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  double worst = 0.0, worst64 = 0.0;
  const int n = 1000000;
  for (int t = 0; t < n; ++t) {
    double u[7];
    const int kind = t % 4;
    const double base = U(g) * std::ldexp(1.0, (int)(200 * U(g)));
    for (int k = 0; k < 7; ++k) {
      if (kind == 0) u[k] = base * (1.0 + 1e-4 * U(g));                    // a smooth field: cancellation
      else if (kind == 1) u[k] = U(g) * std::ldexp(1.0, (int)(40 * U(g))); // mixed magnitudes
      else if (kind == 2) u[k] = (k % 3) ? base * U(g) : 0.0;              // zeros (walls)
      else u[k] = (k & 1) ? -u[0] : base;                                  // ghosts
    }
    long double s = -6.0L * u[0], big = 0.0L;
    double s64 = 0.0;
    for (int k = 0; k < 7; ++k) big = std::max(big, fabsl((long double)u[k]));
    s64 = std::fma(-6.0, u[0], ((u[1] + u[2]) + (u[3] + u[4])) + (u[5] + u[6]));
    for (int k = 1; k < 7; ++k) s += u[k];
    if (big == 0.0L) continue;
    // seven truncations of 2^-57 (the centre's six times) and half an ulp of the result
    const double ulp = (double)(fabsl(s) / big) * std::ldexp(1.0, -53);
    const double err = (double)(fabsl(stencil(u) - s) / big);
    worst = std::max(worst, (err - ulp) * std::ldexp(1.0, 57));
    worst64 = std::max(worst64, (double)(fabsl(s64 - s) / big) * std::ldexp(1.0, 57));
  }
  int edges = 0;
  const double inf = INFINITY, nan = NAN;
  double z[7] = {0, 0, 0, 0, 0, 0, 0};
  edges += stencil(z) != 0.0;
  double a[7] = {1, inf, 0, 0, 0, 0, 0}, b[7] = {1, 2, nan, 0, 0, 0, 0};
  edges += !std::isnan(stencil(a));
  edges += !std::isnan(stencil(b));
  double c[7] = {0, 1, -1, 0x1p-30, 0, 0, 0};
  edges += stencil(c) != 0x1p-30;
  double d[7] = {0, 1e308, 1e308, 0, 0, 0, 0};
  edges += !std::isinf(stencil(d));
  double e[7] = {0, 5e-324, 0, 0, 0, 0, 0};   // subnormal arguments count as zero
  edges += stencil(e) != 0.0;
  // every power-of-two boundary of the conversion back
  int carry = 0;
  for (int k = 1; k < 62; ++k)
    for (int d2 = -1; d2 <= 1; ++d2) {
      const int64_t S = ((int64_t)1 << k) + d2;
      if (S <= 0) continue;
      carry += fix_value(S, 1080) != (double)S;
      carry += fix_value(-S, 1080) != -(double)S;
    }
  std::printf("n %d\nworst_millionths %lld\nworst64_millionths %lld\nedges %d\ncarry %d\n", n, (long long)(worst * 1e6),
              (long long)(worst64 * 1e6), edges, carry);
  return 0;
}
