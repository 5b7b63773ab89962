// Twiddle constants of the register DFTs (plane.cuh), and the jobs and spectral
// weight of the tensor-core transform pass (tc_pass.cuh).
#pragma once

#include "transforms.cuh"

namespace kfbim {

// cos and sin of 2 pi j / 16 for j in 0..15 (exact octant symmetry)
__host__ __device__ constexpr double cos16(int j) {
  constexpr double c1 = 0.92387953251128675613, c2 = 0.70710678118654752440, c3 = 0.38268343236508977173;
  j &= 15;
  return j == 0 ? 1.0 : j == 1 ? c1 : j == 2 ? c2 : j == 3 ? c3 : j == 4 ? 0.0 : j == 5 ? -c3
       : j == 6 ? -c2 : j == 7 ? -c1 : j == 8 ? -1.0 : j == 9 ? -c1 : j == 10 ? -c2 : j == 11 ? -c3
       : j == 12 ? 0.0 : j == 13 ? c3 : j == 14 ? c2 : c1;
}
__host__ __device__ constexpr double sin16(int j) { return cos16(j - 4); }

// cos and sin of 2 pi j / 24 for j in 0..23 (multiples of 15 degrees)
__host__ __device__ constexpr double cos24(int j) {
  constexpr double c15 = 0.96592582628906828675, c30 = 0.86602540378443864676, c45 = 0.70710678118654752440,
                   c60 = 0.5, c75 = 0.25881904510252076235;
  j = ((j % 24) + 24) % 24;
  const int q = j % 12;   // cos(x + 180) = -cos x
  const double v = q == 0 ? 1.0 : q == 1 ? c15 : q == 2 ? c30 : q == 3 ? c45 : q == 4 ? c60 : q == 5 ? c75
                 : q == 6 ? 0.0 : q == 7 ? -c75 : q == 8 ? -c60 : q == 9 ? -c45 : q == 10 ? -c30 : -c15;
  return j < 12 ? v : -v;
}
__host__ __device__ constexpr double sin24(int j) { return cos24(j - 6); }

template <typename T, int N>
__device__ __forceinline__ T spectral_weight2(const PassArgs& a, const T* __restrict__ s2, T inv_mu,
                                              int i, int j, int k) {
  const T sum = s2[a.kind[0] * N + i] + s2[a.kind[1] * N + j] + s2[a.kind[2] * N + k];
  const int ac = a.wc == 0 ? i : (a.wc == 1 ? j : k);
  // correctly rounded reciprocal: the same value as T(1) / sum
  T isum;
  if constexpr (sizeof(T) == 4) isum = __frcp_rn(sum);
  else isum = __drcp_rn(sum);
  if (a.wmode == W_SCHUR) return s2[ac] * isum * inv_mu;
  if (ac == 0) return T(0);
  const T h = T(a.h);
  if (a.wmode == W_POISSON) return h * h * isum * inv_mu;
  return T(-2) * h * sqrt(T(0.25) * s2[ac]) * isum * inv_mu;   // W_RHS
}

// One pass of one field, and up to MAXJ independent passes of a launch.
template <typename Tin, typename Tout>
struct PassJob {
  const Tin* in;
  Tout* out;
  PassArgs a;
};
template <typename Tin, typename Tout, int MAXJ>
struct PassJobs {
  PassJob<Tin, Tout> j[MAXJ];
};

}  // namespace kfbim
