// Host check of k_rhs_moments (kernels.cuh): right-hand sides [f | g] with g a large
// constant and a small rest, zero away from a few cells, and a Navier one (no mean
// removed).  Prints, per case, the relative errors of gmean and ref2 against long-double sums.
#include <cmath>
#include <cstdio>
#include <vector>

#include "kernels.cuh"

using namespace kfbim;

static int run(const char* name, int64_t n3, int stokes, const std::vector<double>& rhs) {
  double *d, *partial, *out;
  unsigned int* ticket;
  const int nb = red_blocks(4 * n3);
  cudaMalloc(&d, rhs.size() * sizeof(double));
  cudaMalloc(&partial, sizeof(double) * MOMENT_DOUBLES * nb);
  cudaMalloc(&out, 2 * sizeof(double));
  cudaMalloc(&ticket, sizeof(unsigned int));
  cudaMemset(ticket, 0, sizeof(unsigned int));
  cudaMemcpy(d, rhs.data(), rhs.size() * sizeof(double), cudaMemcpyHostToDevice);
  k_rhs_moments<<<nb, RED_THREADS>>>(d, n3, stokes, partial, ticket, out, out + 1);
  double got[2] = {0, 0};
  const cudaError_t e = cudaMemcpy(got, out, sizeof(got), cudaMemcpyDeviceToHost);
  cudaFree(d);
  cudaFree(partial);
  cudaFree(out);
  cudaFree(ticket);
  if (e != cudaSuccess) {
    std::fprintf(stderr, "%s\n", cudaGetErrorString(e));
    return 1;
  }
  long double mean = 0, ref = 0;
  for (int64_t k = 0; k < n3; ++k) mean += rhs[3 * n3 + k];
  mean = stokes ? mean / n3 : 0;
  for (int64_t k = 0; k < 3 * n3; ++k) ref += (long double)rhs[k] * rhs[k];
  for (int64_t k = 0; k < n3; ++k) ref += (rhs[3 * n3 + k] - mean) * (rhs[3 * n3 + k] - mean);
  const double em = mean != 0 ? std::fabs((double)((got[0] - mean) / mean)) : std::fabs(got[0]);
  std::printf("%s %.6e %.6e\n", name, em, std::fabs((double)((got[1] - ref) / ref)));
  return 0;
}

int main() {
  int bad = 0;
  for (const int N : {16, 96}) {
    const int64_t n3 = (int64_t)N * N * N;
    std::vector<double> r(4 * n3, 0.0);
    char name[64];
    for (int64_t k = 0; k < n3; ++k) r[3 * n3 + k] = 1e5 + 1e-3 * std::sin(0.37 * (double)k);
    std::snprintf(name, sizeof(name), "constant_%d", N);
    bad |= run(name, n3, 1, r);
    std::snprintf(name, sizeof(name), "navier_%d", N);
    bad |= run(name, n3, 0, r);
    for (int64_t k = 0; k < n3; ++k) r[3 * n3 + k] = k % 97 == 5 ? 1.5 + std::cos(0.11 * (double)k) : 0.0;
    for (int64_t k = 0; k < 3 * n3; ++k) r[k] = k % 53 == 7 ? std::sin(0.7 * (double)k) : 0.0;
    std::snprintf(name, sizeof(name), "interface_%d", N);
    bad |= run(name, n3, 1, r);
  }
  return bad;
}
