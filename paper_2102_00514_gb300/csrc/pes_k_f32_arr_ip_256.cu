// Persistent smoother kernel: float, the given arrays in place, 256 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(float, pes::KK_ARRAYS_IN_PLACE, 256)
