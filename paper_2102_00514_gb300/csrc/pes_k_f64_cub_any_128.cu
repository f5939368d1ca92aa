// Persistent smoother kernel: double, cubature / unscented, any model, 128 threads per block.
#include "pes_launch_impl.cuh"
PES_INSTANTIATE(double, pes::KK_CUBATURE_ANY, 128)
