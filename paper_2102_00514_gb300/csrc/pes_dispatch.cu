// Dispatch from run-time (precision, linearisation, block size) to the
// compiled configurations of the persistent kernel.
#include <algorithm>

#include "pes_internal.h"

namespace pes {

template <typename T, int NT>
static cudaError_t launch_nt(const KParams<T>& p, int lin, int nb, cudaStream_t st)
{
    const bool ct = p.model.kind == MODEL_CT_BEARINGS;
    if constexpr (sizeof(T) == 4 && NT == 256)   // the one compiled form (filter_in_place, smooth_in_place)
        if (lin == LIN_ARRAYS && p.in_place) return launch_cfg<T, KK_ARRAYS_IN_PLACE, NT>(p, nb, st);
    if (p.in_place) return cudaErrorInvalidValue;
    if (lin == LIN_ARRAYS) return launch_cfg<T, KK_ARRAYS, NT>(p, nb, st);
    if (lin == LIN_IEKS) return ct ? launch_cfg<T, KK_IEKS, NT>(p, nb, st) : launch_cfg<T, KK_IEKS_ANY, NT>(p, nb, st);
    if (lin == LIN_GH) return launch_cfg<T, KK_GH, NT>(p, nb, st);
    return ct ? launch_cfg<T, KK_CUBATURE, NT>(p, nb, st) : launch_cfg<T, KK_CUBATURE_ANY, NT>(p, nb, st);
}

// The model is not known here: the smaller capacity of the two forms.
template <typename T, int NT>
static int capacity_nt(int lin, int device)
{
    if (lin == LIN_ARRAYS) {
        const int n = capacity_cfg<T, KK_ARRAYS, NT>(device);
        if constexpr (sizeof(T) == 4 && NT == 256) return std::min(n, capacity_cfg<T, KK_ARRAYS_IN_PLACE, NT>(device));
        return n;
    }
    if (lin == LIN_GH) return capacity_cfg<T, KK_GH, NT>(device);
    const int a = lin == LIN_IEKS ? capacity_cfg<T, KK_IEKS, NT>(device) : capacity_cfg<T, KK_CUBATURE, NT>(device);
    const int b = lin == LIN_IEKS ? capacity_cfg<T, KK_IEKS_ANY, NT>(device) : capacity_cfg<T, KK_CUBATURE_ANY, NT>(device);
    return a < b ? a : b;
}

cudaError_t launch_persistent(const KParams<float>& p, int lin, int nt, int nb, cudaStream_t st)
{
    if (nt == 256) return launch_nt<float, 256>(p, lin, nb, st);
    if (nt == 128) return launch_nt<float, 128>(p, lin, nb, st);
    return cudaErrorInvalidValue;
}

cudaError_t launch_persistent(const KParams<double>& p, int lin, int nt, int nb, cudaStream_t st)
{
    if (nt == 128) return launch_nt<double, 128>(p, lin, nb, st);
    return cudaErrorInvalidValue;
}

int coop_capacity(float, int lin, int nt, int device)
{
    if (nt == 256) return capacity_nt<float, 256>(lin, device);
    if (nt == 128) return capacity_nt<float, 128>(lin, device);
    return 0;
}

int coop_capacity(double, int lin, int nt, int device)
{
    if (nt == 128) return capacity_nt<double, 128>(lin, device);
    return 0;
}

bool nt_supported(float, int nt) { return nt == 128 || nt == 256; }
bool nt_supported(double, int nt) { return nt == 128; }

}  // namespace pes
