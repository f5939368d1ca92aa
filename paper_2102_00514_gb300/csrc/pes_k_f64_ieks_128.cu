// Persistent smoother kernel: double, Taylor, coordinated turn, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(double, pes::KK_IEKS, 128)
