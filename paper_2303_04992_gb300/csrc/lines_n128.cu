// The one-axis transform kernels for N = 128 (lines.h).
#include "lines_impl.cuh"

KFBIM_LINES_INSTANTIATE(128)
