// The one-axis transform kernels for N = 96 (lines.h).
#include "lines_impl.cuh"

KFBIM_LINES_INSTANTIATE(96)
