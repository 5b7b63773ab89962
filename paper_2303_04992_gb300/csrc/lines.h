// Host entry of the one-axis transform pass of lines.cuh.  Each grid size's
// kernels are instantiated in a translation unit of their own (lines_n32.cu ...
// lines_n256.cu) so that they compile in parallel.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include "lines.cuh"

namespace kfbim {

// Jobs per launch: 3 for one instance, 48 for a batch of 16 instances.
constexpr int kLineJobs = 3;
constexpr int kLineBatchJobs = 48;

// Raises a kernel's dynamic shared-memory limit on the current device once.
cudaError_t raise_dynamic_smem(const void* kern, size_t bytes);

// One launch of operation op (lines::Op) for grid N over njobs jobs (blockIdx.y =
// job), with the FP32 or FP64 tables of the context.  (Tin, T, Tout) =
// (double, double, double) with MAXJ = 3; (float, float, float) and, for
// op = OP_F2 only, (double, float, float), for OP_I2 only, (float, float, double),
// with MAXJ = 3 and kLineBatchJobs;
// cudaErrorInvalidValue for a combination that has no kernel (plain DST-I passes
// of a batch).
template <int N, typename Tin, typename T, typename Tout, int MAXJ>
cudaError_t lines_launch(int op, const lines::Jobs<Tin, Tout, MAXJ>& jobs, int njobs, const lines::Scales<T>& sc,
                         const C2<T>* tw, const C2<T>* qN, const T* s2, cudaStream_t s);

}  // namespace kfbim
