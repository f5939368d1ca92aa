// Persistent smoother kernel: float, Gauss-Hermite, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(float, pes::KK_GH, 128)
