// Persistent smoother kernel: float, the given arrays, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(float, pes::KK_ARRAYS, 128)
