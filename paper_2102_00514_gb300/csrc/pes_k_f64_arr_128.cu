// Persistent smoother kernel: double, the given arrays, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(double, pes::KK_ARRAYS, 128)
