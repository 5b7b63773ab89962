// The one-axis transform kernels for N = 256 (lines.h).
#include "lines_impl.cuh"

KFBIM_LINES_INSTANTIATE(256)
