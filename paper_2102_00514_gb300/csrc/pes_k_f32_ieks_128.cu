// Persistent smoother kernel: float, Taylor, coordinated turn, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(float, pes::KK_IEKS, 128)
