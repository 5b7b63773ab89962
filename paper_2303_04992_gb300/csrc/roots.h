// Roots of unity for the transform tables.  Plain C++: the CPU test suite compiles
// this header with g++ and compares the roots with long-double ones.
#pragma once

#include <cmath>

namespace kfbim {

// exp(-i pi k / n) for 0 <= k < 2 n, by symmetry from an angle of at most pi / 4, whose
// rounding is then 2e-16 at most: cos and sin of a rounded angle of up to 2 pi are 9.7e-16
// off, which an FP64 Poisson solve sees (6.0e-16 of error at N = 96, 4.6e-16 with these).
inline void unit_root(int k, int n, double* re, double* im) {
  const bool up = k > n;            // lower half circle to the upper one
  if (up) k = 2 * n - k;
  const bool left = 2 * k > n;      // second quadrant to the first
  if (left) k = n - k;
  const bool swap = 4 * k > n;      // second octant to the first
  const double a = swap ? M_PI * (n - 2 * k) / (2.0 * n) : M_PI * k / (double)n;
  const double c = std::cos(a), s = std::sin(a);
  *re = left ? -(swap ? s : c) : (swap ? s : c);
  *im = up ? (swap ? c : s) : -(swap ? c : s);
}

}  // namespace kfbim
