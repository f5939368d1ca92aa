// Persistent smoother kernel: float, Taylor, any model, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(float, pes::KK_IEKS_ANY, 128)
