// Device side of the Levenberg-Marquardt iteration with adaptive damping
// (Sec. 3 names the LM variant of the IEKS; the host loop is
// pes_ieks_run_lm in pes_api.cu): the change of every trajectory's MAP objective
// by a step, the per-trajectory accept/reject decision and damping update, and
// the restore of a rejected trajectory's nominal.
//
// The change is summed over the states as it is, in FP64 for either precision,
// and not as the difference of two objectives: near convergence a step of relative
// size 1e-8 changes the objective by 1e-16 of it, and whether two rounded sums
// compare as smaller would hang on the order of their additions. With a residual e
// and its change D, a term's change is 1/2 D^T W (2 e + D); D is formed from the
// state's change without cancellation (f_change, obs_change). Steps of relative
// size 1e-9 (a change of 1e-19 of the objective) are then still told apart.
#include "pes_internal.h"
#include "pes_lm.cuh"

namespace pes {

namespace {

PES_DEV int traj_of_k(const int64_t* off, int B, int64_t k)
{
    int lo = 0, hi = B - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(off + mid) <= k) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// sincos, by its series (to 1e-19) for the small angles that a step turns by
PES_DEV void sincos_of_small(double x, double* s, double* c)
{
    if (fabs(x) < 0.05) {
        const double x2 = x * x;
        *s = x * (1.0 - x2 * (1.0 / 6.0 - x2 * (1.0 / 120.0 - x2 * (1.0 / 5040.0 - x2 * (1.0 / 362880.0)))));
        *c = 1.0 - x2 * (0.5 - x2 * (1.0 / 24.0 - x2 * (1.0 / 720.0 - x2 * (1.0 / 40320.0 - x2 * (1.0 / 3628800.0)))));
    } else {
        sincos(x, s, c);
    }
}

// wrap_angle, without its quotient where the angle is on the branch already
PES_DEV double wrap_near(double a) { return fabs(a) < 3.14 ? a : wrap_angle(a); }

// x - f(xp) and its change by the steps d of x and dp of xp, in FP64
PES_DEV void f_change(const LMParams& p, const double* x, const double* d, const double* xp, const double* dp, double* e,
                      double* de)
{
    if (p.kind == MODEL_LINEAR) {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            double s = p.c[i], t = 0.0;
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                s = fma(p.F[i * 5 + l], xp[l], s);
                t = fma(p.F[i * 5 + l], dp[l], t);
            }
            e[i] = x[i] - s;
            de[i] = d[i] - t;
        }
        return;
    }
    // Sines and cosines of the old and the new angle and their changes, all from those
    // of the mean angle and of half the change: the FP64 pipe takes 64 cycles for every
    // instruction of a warp, so a sincos or a quotient less counts.
    const double dt = p.dt, w = xp[4], dw = dp[4], wn = w + dw;
    const double a = w * dt, an = wn * dt, da = dw * dt, half = 0.5 * da;
    double sh, ch, sm, cm;
    sincos_of_small(half, &sh, &ch);
    sincos_of_small(a + half, &sm, &cm);
    CTCoef<double> k, n;
    k.s = sm * ch - cm * sh;
    k.c = cm * ch + sm * sh;
    n.s = sm * ch + cm * sh;
    n.c = cm * ch - sm * sh;
    const double dc = -2.0 * sm * sh, ds = 2.0 * cm * sh;
    // A1 = sin(w dt) / w, A2 = (1 - cos(w dt)) / w and their changes
    double dA1, dA2;
    if (fabs(a) < 0.01 && fabs(an) < 0.01) {   // ct_coef's series
        const double a2 = a * a, an2 = an * an, s2 = a2 + an2, m = a * an;
        k.A1 = dt * (1.0 - a2 * (1.0 / 6.0) + a2 * a2 * (1.0 / 120.0));
        k.A2 = dt * a * (0.5 - a2 * (1.0 / 24.0) + a2 * a2 * (1.0 / 720.0));
        dA1 = dt * da * (a + an) * (s2 * (1.0 / 120.0) - 1.0 / 6.0);
        dA2 = dt * da * (0.5 - (s2 + m) * (1.0 / 24.0) + (s2 * s2 - m * m + m * s2) * (1.0 / 720.0));
        n.A1 = k.A1 + dA1;
        n.A2 = k.A2 + dA2;
    } else {
        k = ct_coef(w, dt);
        n = ct_coef(wn, dt);
        if (fabs(da) <= 0.5 * fabs(a)) {
            dA1 = (ds - k.A1 * dw) / wn;
            dA2 = (-dc - k.A2 * dw) / wn;
        } else {
            dA1 = n.A1 - k.A1;
            dA2 = n.A2 - k.A2;
        }
    }
    double inc[5];
    ct_increment(xp, k, inc);
    e[0] = (x[0] - xp[0]) - inc[0];
    e[1] = (x[1] - xp[1]) - inc[1];
#pragma unroll
    for (int i = 2; i < 5; ++i) e[i] = x[i] - inc[i];
    de[0] = (d[0] - dp[0]) - (n.A1 * dp[2] - n.A2 * dp[3] + dA1 * xp[2] - dA2 * xp[3]);
    de[1] = (d[1] - dp[1]) - (n.A2 * dp[2] + n.A1 * dp[3] + dA2 * xp[2] + dA1 * xp[3]);
    de[2] = d[2] - (n.c * dp[2] - n.s * dp[3] + dc * xp[2] - ds * xp[3]);
    de[3] = d[3] - (n.s * dp[2] + n.c * dp[3] + ds * xp[2] + dc * xp[3]);
    de[4] = d[4] - dp[4];
}

// y - h(x) and its change by the step d of x. Bearings (residuals on the branch nearest
// zero): r holds the residuals before the step, which are kept from step to step, and
// the change is the angle between the old and the new line of sight; two arctangents
// less per state, 264 -> 209 us at 300,001 states.
PES_DEV void obs_change(const LMParams& p, int b, const double* x, const double* d, const double* y, double* r,
                        double* dr)
{
    if (p.kind == MODEL_LINEAR) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            double s = p.d[i], t = 0.0;
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                s = fma(p.H[i * 5 + l], x[l], s);
                t = fma(p.H[i * 5 + l], d[l], t);
            }
            r[i] = y[i] - s;
            dr[i] = -t;
        }
        return;
    }
    const double* s = p.sensors + (p.sensors_per_traj ? 4 * b : 0);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const double rx = x[0] - s[2 * i], ry = x[1] - s[2 * i + 1];
        const double cross = rx * d[1] - ry * d[0], dot = rx * (rx + d[0]) + ry * (ry + d[1]);
        double turn;
        if (fabs(cross) < 0.01 * dot) {   // its series, to 1e-19
            const double q = cross / dot, q2 = q * q;
            turn = q * (1.0 - q2 * (1.0 / 3.0 - q2 * (0.2 - q2 * (1.0 / 7.0 - q2 * (1.0 / 9.0)))));
        } else {
            turn = atan2(cross, dot);
        }
        const double rn = wrap_near(r[i] - turn);
        dr[i] = rn == r[i] - turn ? -turn : rn - r[i];   // else it crosses to another branch
    }
}

// 1/2 de^T S (2 e + de), S symmetric packed
template <int N>
PES_DEV double quad_change(const double* S, const double* e, const double* de)
{
    double h[N], q = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) h[i] = fma(0.5, de[i], e[i]);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        double v = 0.0;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int a = i < j ? i : j, c = i < j ? j : i;
            v = fma(S[N == 5 ? si(a, c) : si2(a, c)], h[j], v);
        }
        q = fma(de[i], v, q);
    }
    return q;
}

// Contiguous runs of lanes that hold the same trajectory add their values
// into the run's first lane, which adds them to the trajectory's accumulator.
// Every lane of the warp calls (b < 0: a lane without a state, nothing added).
PES_DEV void warp_segment_add(double v, int b, double* acc)
{
    const unsigned grp = __match_any_sync(0xffffffffu, b);
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double o = __shfl_down_sync(0xffffffffu, v, off);
        const int src = lane + off;
        if (src < 32 && ((grp >> src) & 1u)) v += o;
    }
    if (b >= 0 && lane == __ffs(grp) - 1) atomicAdd(acc + b, v);
}

}  // namespace

// The bearings' residuals at the nominal x, into p.resid (a trajectory's first state
// has none).
template <typename T>
__global__ void lm_resid_kernel(const LMParams p, const T* x, const T* y)
{
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (ix >= p.cs) return;
    const int s = (int)(ix / p.NL);
    const int64_t k = (ix - (int64_t)s * p.NL) * p.L + s;
    if (k >= p.N) return;
    const int b = traj_of_k(p.offsets, p.B, k);
    if (k == __ldg(p.offsets + b)) return;
    const double* q = p.sensors + (p.sensors_per_traj ? 4 * b : 0);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        p.resid[i * p.cs + ix] = wrap_near((double)y[i * p.cs + ix] -
                                           atan2((double)x[p.cs + ix] - q[2 * i + 1], (double)x[ix] - q[2 * i]));
}

// What the step from xold to x (both in the smoother kernel's lane-major slots)
// changes every trajectory's MAP objective by, added into p.change; also the
// squared step into p.num and ||x||^2 into p.den if the tolerance asks for them.
template <typename T>
__global__ void lm_change_kernel(const LMParams p, const T* x, const T* xold, const T* y, const T* m0, const T* P0)
{
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool valid = ix < p.cs;
    int64_t k = 0;
    int s = 0, lane = 0;
    if (valid) {
        s = (int)(ix / p.NL);
        lane = (int)(ix - (int64_t)s * p.NL);
        k = (int64_t)lane * p.L + s;
        valid = k < p.N;
    }
    // every lane stays to the warp's reductions; one without a state adds nothing
    const int b = valid ? traj_of_k(p.offsets, p.B, k) : -1;
    double dJ = 0.0, num = 0.0, den = 0.0;
    if (valid) {
        double xo[5], d[5];
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            const double xn = (double)x[c * p.cs + ix];
            xo[c] = (double)xold[c * p.cs + ix];
            d[c] = xn - xo[c];
            if (p.norms) {
                num = fma(d[c], d[c], num);
                den = fma(xn, xn, den);
            }
        }
        if (k == __ldg(p.offsets + b)) {
            // prior: 1/2 |L^{-1} (x_0 - m0)|^2, P0 = L L^T
            double P[15], Lc[25], rd[5], z[5], dz[5];
#pragma unroll
            for (int c = 0; c < 15; ++c) P[c] = (double)P0[15 * b + c];
            chol_pd(P, Lc, rd);
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                double t = xo[i] - (double)m0[5 * b + i], u = d[i];
#pragma unroll
                for (int l = 0; l < i; ++l) {
                    t = fma(-Lc[i * 5 + l], z[l], t);
                    u = fma(-Lc[i * 5 + l], dz[l], u);
                }
                z[i] = t * rd[i];
                dz[i] = u * rd[i];
                dJ = fma(dz[i], fma(0.5, dz[i], z[i]), dJ);
            }
        } else {
            const int64_t ixp = s > 0 ? ix - p.NL : (int64_t)(p.L - 1) * p.NL + (lane - 1);
            double xp[5], dp[5], e[5], de[5];
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                xp[c] = (double)xold[c * p.cs + ixp];
                dp[c] = (double)x[c * p.cs + ixp] - xp[c];
            }
            f_change(p, xo, d, xp, dp, e, de);
            dJ = quad_change<5>(p.Qi, e, de);
            double yk[2], r[2], dr[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                yk[i] = (double)y[i * p.cs + ix];
                r[i] = p.resid[i * p.cs + ix];
            }
            obs_change(p, b, xo, d, yk, r, dr);
            dJ += quad_change<2>(p.Ri, r, dr);
#pragma unroll
            for (int i = 0; i < 2; ++i) p.resid_step[i * p.cs + ix] = r[i] + dr[i];
        }
    }
    warp_segment_add(dJ, b, p.change);
    if (!p.norms) return;
    warp_segment_add(num, b, p.num);
    warp_segment_add(den, b, p.den);
}

// Per trajectory: keep the step if it lowered the objective (damping / nu),
// else keep the nominal (damping * nu); record convergence (the step's
// relative size <= tol) and count the trajectories still unconverged.
template <typename T>
__global__ void lm_decide_kernel(const LMParams p, T* lam, int it, double tol, double nu)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= p.B) return;
    const double num = p.num[b], den = p.den[b];
    const double rel = den > 0.0 ? sqrt(num / den) : sqrt(num);
    if (p.change[b] < 0.0) {
        lam[b] = (T)((double)lam[b] / nu);
        p.accepted[b] += 1;
        p.reject[b] = 0;
    } else {
        lam[b] = (T)((double)lam[b] * nu);
        p.reject[b] = 1;
    }
    if (tol > 0.0 && p.conv_iter[b] == 0 && rel <= tol) p.conv_iter[b] = it;
    if (p.conv_iter[b] == 0) atomicAdd(p.unconv, 1);
}

// A rejected trajectory's nominal and covariances go back to their values before the
// step; the others' residuals become those after it.
template <typename T>
__global__ void lm_restore_kernel(const LMParams p, T* x, T* P, const T* xold, const T* Pold)
{
    const int64_t ix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (ix >= p.cs) return;
    const int s = (int)(ix / p.NL);
    const int lane = (int)(ix - (int64_t)s * p.NL);
    const int64_t k = (int64_t)lane * p.L + s;
    if (k >= p.N) return;
    const int b = traj_of_k(p.offsets, p.B, k);
    if (!p.reject[b]) {
#pragma unroll
        for (int i = 0; i < 2; ++i) p.resid[i * p.cs + ix] = p.resid_step[i * p.cs + ix];
        return;
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) x[c * p.cs + ix] = xold[c * p.cs + ix];
#pragma unroll
    for (int c = 0; c < 15; ++c) P[c * p.cs + ix] = Pold[c * p.cs + ix];
}

template <typename T>
__global__ void lm_fill_kernel(T* lam, int B, double v)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) lam[b] = (T)v;
}

template <typename T>
cudaError_t launch_lm_resid(const LMParams& p, const T* x, const T* y, cudaStream_t st)
{
    if (p.kind == MODEL_LINEAR) return cudaSuccess;
    lm_resid_kernel<T><<<(unsigned)((p.cs + 255) / 256), 256, 0, st>>>(p, x, y);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_lm_change(const LMParams& p, const T* x, const T* xold, const T* y, const T* m0, const T* P0,
                             cudaStream_t st)
{
    const unsigned blocks = (unsigned)((p.cs + 255) / 256);
    lm_change_kernel<T><<<blocks, 256, 0, st>>>(p, x, xold, y, m0, P0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_lm_decide(const LMParams& p, T* lam, int it, double tol, double nu, cudaStream_t st)
{
    lm_decide_kernel<T><<<(p.B + 127) / 128, 128, 0, st>>>(p, lam, it, tol, nu);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_lm_restore(const LMParams& p, T* x, T* P, const T* xold, const T* Pold, cudaStream_t st)
{
    const unsigned blocks = (unsigned)((p.cs + 255) / 256);
    lm_restore_kernel<T><<<blocks, 256, 0, st>>>(p, x, P, xold, Pold);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_lm_fill(T* lam, int B, double v, cudaStream_t st)
{
    lm_fill_kernel<T><<<(B + 127) / 128, 128, 0, st>>>(lam, B, v);
    return cudaGetLastError();
}

#define PES_LM_INSTANTIATE(T)                                                                                     \
    template cudaError_t launch_lm_resid<T>(const LMParams&, const T*, const T*, cudaStream_t);                   \
    template cudaError_t launch_lm_change<T>(const LMParams&, const T*, const T*, const T*, const T*, const T*,   \
                                             cudaStream_t);                                                       \
    template cudaError_t launch_lm_decide<T>(const LMParams&, T*, int, double, double, cudaStream_t);           \
    template cudaError_t launch_lm_restore<T>(const LMParams&, T*, T*, const T*, const T*, cudaStream_t);       \
    template cudaError_t launch_lm_fill<T>(T*, int, double, cudaStream_t);
PES_LM_INSTANTIATE(float)
PES_LM_INSTANTIATE(double)

}  // namespace pes
