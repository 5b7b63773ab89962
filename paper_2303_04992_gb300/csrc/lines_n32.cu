// The one-axis transform kernels for N = 32 (lines.h).
#include "lines_impl.cuh"

KFBIM_LINES_INSTANTIATE(32)
