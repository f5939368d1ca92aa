// Parameters of the Levenberg-Marquardt kernels (pes_lm.cu): the model in
// FP64 (the objective's change is evaluated in FP64 for either precision), the
// lane-major geometry of the smoother kernel, and per-trajectory accumulators.
#pragma once

#include "pes_model.cuh"

namespace pes {

struct LMParams {
    int64_t N;
    const int64_t* offsets;
    int B;
    int L, NL;
    int64_t cs;
    int kind;
    int sensors_per_traj;
    double dt;
    const double* sensors;   // device [1 or B][4]
    double F[25], c[5], H[10], d[2];   // linear model
    double Qi[15], Ri[3];              // inverses of Q and R (packed)
    double* resid;      // [2][cs] the bearings' residuals at the nominal
    double* resid_step; // [2][cs] and after the step
    double* change;     // [B] what the step changes the objective by
    int norms;          // whether the two that follow are wanted
    double* num;        // [B] squared step
    double* den;        // [B] squared norm after it
    int* reject;        // [B]
    int* accepted;      // [B] steps accepted so far
    int* conv_iter;     // [B] first converged iteration (0: none)
    int* unconv;        // trajectories not yet converged
};

// The bearings' residuals at the first nominal x into p.resid (a linear model needs none).
template <typename T>
cudaError_t launch_lm_resid(const LMParams& p, const T* x, const T* y, cudaStream_t st);
// What the step from xold to x changes every trajectory's objective by, the
// squared step and the squared norm after it, added into p.change, p.num, p.den.
template <typename T>
cudaError_t launch_lm_change(const LMParams& p, const T* x, const T* xold, const T* y, const T* m0, const T* P0,
                             cudaStream_t st);
template <typename T>
cudaError_t launch_lm_decide(const LMParams& p, T* lam, int it, double tol, double nu, cudaStream_t st);
template <typename T>
cudaError_t launch_lm_restore(const LMParams& p, T* x, T* P, const T* xold, const T* Pold, cudaStream_t st);
template <typename T>
cudaError_t launch_lm_fill(T* lam, int B, double v, cudaStream_t st);

}  // namespace pes
