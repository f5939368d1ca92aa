// Persistent smoother kernel: float, cubature / unscented, coordinated turn, 256 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(float, pes::KK_CUBATURE, 256)
