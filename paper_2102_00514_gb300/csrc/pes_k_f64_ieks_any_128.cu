// Persistent smoother kernel: double, Taylor, any model, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(double, pes::KK_IEKS_ANY, 128)
