// Definition of lines_launch (lines.h), included by the per-grid-size
// translation units only.
#pragma once

#include "lines.h"

namespace kfbim {

template <int N, int OP, typename Tin, typename T, typename Tout, int MAXJ>
cudaError_t lines_launch_op(const lines::Jobs<Tin, Tout, MAXJ>& jobs, int njobs, const lines::Scales<T>& sc,
                            const C2<T>* tw, const C2<T>* qN, const T* s2, cudaStream_t s) {
  using L = lines::LShape<N, T>;
  auto kern = lines::k_lines<Tin, T, Tout, N, OP, MAXJ>;
  const cudaError_t e = raise_dynamic_smem(reinterpret_cast<const void*>(kern), L::bytes);
  if (e != cudaSuccess) return e;
  return launch_overlapped(sizeof(T) == 4 && N <= 128, kern, dim3((unsigned)L::BLOCKS, (unsigned)njobs), L::THREADS,
                           L::bytes, s, jobs, sc, tw, qN, s2);
}

template <int N, typename Tin, typename T, typename Tout, int MAXJ>
cudaError_t lines_launch(int op, const lines::Jobs<Tin, Tout, MAXJ>& jobs, int njobs, const lines::Scales<T>& sc,
                         const C2<T>* tw, const C2<T>* qN, const T* s2, cudaStream_t s) {
#define KFBIM_LINES_OP(OP) \
  case OP: return lines_launch_op<N, OP, Tin, T, Tout, MAXJ>(jobs, njobs, sc, tw, qN, s2, s)
  if constexpr (sizeof(Tout) > sizeof(T)) {
    switch (op) {
      KFBIM_LINES_OP(lines::OP_I2);
      default: break;
    }
  } else if constexpr (sizeof(Tin) == sizeof(T)) {
    switch (op) {
      KFBIM_LINES_OP(lines::OP_F2);
      KFBIM_LINES_OP(lines::OP_I2);
      KFBIM_LINES_OP(lines::OP_F2I2);
      KFBIM_LINES_OP(lines::OP_F1I1);
      KFBIM_LINES_OP(lines::OP_F1I2);
      default: break;
    }
    if constexpr (MAXJ == kLineJobs && sizeof(T) == 4) {
      switch (op) {   // plain DST-I passes: only through the transform entry point
        KFBIM_LINES_OP(lines::OP_F1);
        KFBIM_LINES_OP(lines::OP_I1);
        default: break;
      }
    }
  } else {
    switch (op) {
      KFBIM_LINES_OP(lines::OP_F2);
      default: break;
    }
  }
#undef KFBIM_LINES_OP
  return cudaErrorInvalidValue;
}

}  // namespace kfbim

#define KFBIM_LINES_INSTANTIATE_ONE(N, TIN, T, TOUT, MAXJ)                                                    \
  template cudaError_t kfbim::lines_launch<N, TIN, T, TOUT, MAXJ>(                                            \
      int, const kfbim::lines::Jobs<TIN, TOUT, MAXJ>&, int, const kfbim::lines::Scales<T>&,                 \
      const kfbim::C2<T>*, const kfbim::C2<T>*, const T*, cudaStream_t);
#define KFBIM_LINES_INSTANTIATE(N)                                                  \
  KFBIM_LINES_INSTANTIATE_ONE(N, double, double, double, kfbim::kLineJobs)          \
  KFBIM_LINES_INSTANTIATE_ONE(N, double, float, float, kfbim::kLineJobs)            \
  KFBIM_LINES_INSTANTIATE_ONE(N, double, float, float, kfbim::kLineBatchJobs)       \
  KFBIM_LINES_INSTANTIATE_ONE(N, float, float, double, kfbim::kLineJobs)            \
  KFBIM_LINES_INSTANTIATE_ONE(N, float, float, double, kfbim::kLineBatchJobs)       \
  KFBIM_LINES_INSTANTIATE_ONE(N, float, float, float, kfbim::kLineJobs)             \
  KFBIM_LINES_INSTANTIATE_ONE(N, float, float, float, kfbim::kLineBatchJobs)
