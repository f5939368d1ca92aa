// Persistent smoother kernel: float, Gauss-Hermite, 256 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(float, pes::KK_GH, 256)
