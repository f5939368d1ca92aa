// Persistent smoother kernel: double, Gauss-Hermite, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(double, pes::KK_GH, 128)
