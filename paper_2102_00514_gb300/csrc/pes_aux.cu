// Element-wise kernels around the persistent smoother: offsets validation,
// nominal initialisation and the stand-alone linearisation (Eqs. 7-10).
#include <algorithm>

#include "pes_internal.h"

namespace pes {

// Grid-stride over the B gaps; any malformed entry raises ST_BADARG.
__global__ void validate_offsets_kernel(const int64_t* offsets, int B, int64_t N, int* status)
{
    const int stride = gridDim.x * blockDim.x;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += stride) {
        const int64_t lo = offsets[b], hi = offsets[b + 1];
        bool bad = !(hi > lo);
        if (b == 0 && lo != 0) bad = true;
        if (b == B - 1 && hi != N) bad = true;
        if (bad) atomicOr(status, ST_BADARG);
    }
}

cudaError_t launch_validate_offsets(const int64_t* offsets, int B, int64_t N, int* status, cudaStream_t st)
{
    const int threads = 256;
    const int blocks = (int)std::min<int64_t>((B + threads - 1) / threads, 4096);
    validate_offsets_kernel<<<blocks, threads, 0, st>>>(offsets, B, N, status);
    return cudaGetLastError();
}

// One thread per state: locate its trajectory by binary search.
PES_DEV int traj_of(const int64_t* offsets, int B, int64_t k)
{
    int lo = 0, hi = B - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(offsets + mid) <= k) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <typename T>
__global__ void convert_kernel(const double* in, T* out, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = T(in[i]);
}

template <typename T>
cudaError_t launch_convert(const double* in, T* out, int n, cudaStream_t st)
{
    const int threads = 256;
    const int blocks = std::max(1, std::min((n + threads - 1) / threads, 1024));
    convert_kernel<T><<<blocks, threads, 0, st>>>(in, out, n);
    return cudaGetLastError();
}

template <typename Ti, typename To>
__global__ void convert_ff_kernel(const Ti* in, To* out, int64_t n)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = To(in[i]);
}

template <typename Ti, typename To>
cudaError_t launch_convert_ff(const Ti* in, To* out, int64_t n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const int threads = 256;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, 152 * 16));
    convert_ff_kernel<Ti, To><<<blocks, threads, 0, st>>>(in, out, n);
    return cudaGetLastError();
}

template cudaError_t launch_convert_ff<float, double>(const float*, double*, int64_t, cudaStream_t);
template cudaError_t launch_convert_ff<double, float>(const double*, float*, int64_t, cudaStream_t);

template cudaError_t launch_convert<float>(const double*, float*, int, cudaStream_t);
template cudaError_t launch_convert<double>(const double*, double*, int, cudaStream_t);

// Caller layout [nc][N] <-> the kernel's lane-major layout [nc][L][NL], where
// state k = lane * L + s sits at s * NL + lane, for several arrays in one
// launch (their components consecutive on the lane-major side).
//
// Bound by memory latency and by instructions: what counts is bytes in flight and
// how few instructions a value takes. A block takes G lanes of some components: with L
// <= W steps a component's states are one contiguous run of the caller's array, so
// both sides are read and written in full lines whatever L is, and a place's index
// serves all the block's components; longer chunks are cut into pieces of W steps, a
// warp reading a lane's piece. Everything a block reads is in flight at once, copied
// into the tile by cp.async, and its stores do not wait. The tile's rows are steps,
// as far apart as keeps the banks free of conflicts on both sides (mv_row). (32 x 32
// tiles of (lane, step) leave columns empty and start every row off a line's boundary:
// the 20 components of 2^20 states, L = 27, took 62 us, one component's index at a
// time 40, here 31; 62 components of 262,144 states, L = 8, 41 -> 23, 20 back 16 ->
// 11; 20 of 5.2 million, L = 134, 211 -> 188.)
constexpr int MV_W = 63, MV_THREADS = 256, MV_NC = 65, MV_BYTES = 47 * 1024;
template <typename T>
constexpr int MV_G = sizeof(T) == 4 ? 128 : 64;

template <typename T>
PES_DEV void copy_async(T* dst, const T* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(sizeof(T)) : "memory");
}

// Words from a row of the tile to the next. The caller's side goes through the tile
// by consecutive states, so that a warp (doubles: half a warp) touches several rows
// of several lanes if a lane has fewer steps than that: rows are as many banks apart.
template <typename T>
__host__ __device__ constexpr int mv_row(int w)
{
    constexpr int n = 128 / sizeof(T);   // words that the banks hold
    return MV_G<T> + (w < n ? (n + w - 1) / w : 1);
}

template <typename T, bool TO_LANES, bool BLOCKED>
__global__ void __launch_bounds__(MV_THREADS) lanes_move_kernel(const __grid_constant__ LaneArrays<T> a, T* lanes,
                                                                int64_t N, int L, int NL, int nc, int per_block)
{
    constexpr int G = MV_G<T>;
    extern __shared__ __align__(16) unsigned char mv_raw[];
    T* tiles = reinterpret_cast<T*>(mv_raw);
    const int64_t cs = (int64_t)L * NL;
    const int l0 = blockIdx.x * G, s0 = blockIdx.y * MV_W;
    const int w = min(MV_W, L - s0), g = min(G, NL - l0), RS = mv_row<T>(w);
    const int64_t k0 = (int64_t)l0 * L + s0;
    const int64_t left = N - k0;   // states from k0 on
    const int t = threadIdx.x;
    const int c0 = blockIdx.z * per_block, c1 = min(nc, c0 + per_block);
    // f(word of the tile, place in the caller's array from k0 on)
    auto caller_side = [&](auto f) {
        if (w == L) {
            const int n = (int)min((int64_t)g * w, left);
            const int dl = MV_THREADS / w, dr = MV_THREADS - dl * w;
            const int di = dr * RS + dl, wrap = 1 - w * RS;
            int r = t % w, i = r * RS + t / w;
            for (int q = t; q < n; q += MV_THREADS) {
                f(i, q);
                r += dr;
                i += di;
                if (r >= w) r -= w, i += wrap;
            }
        } else {
            for (int l = t >> 5; l < g; l += MV_THREADS / 32)
                for (int r = t & 31; r < w; r += 32)
                    if ((int64_t)l * L + r < left) f(r * RS + l, (int64_t)l * L + r);
        }
    };
    // f(word of the tile, place among the component's lane-major values from (s0, l0) on)
    auto lane_side = [&](auto f) {
        const int l = t % G;
        const int64_t most = left - (int64_t)l * L;   // steps from s0 on that the lane has
        const int64_t row = BLOCKED ? nc * 32 : NL;
        const int64_t at = BLOCKED ? (int64_t)(l >> 5) * L * row + (l & 31) : l;
        if (l < g) {
            const int n = (int)min((int64_t)w, most);
            int64_t ix = t / G * row + at;
            int i = t / G * RS + l;
            for (int r = t / G; r < n; r += MV_THREADS / G, ix += MV_THREADS / G * row, i += MV_THREADS / G * RS) f(i, ix);
        }
    };
    const int nb = c1 - c0, tile = w * RS;
    __shared__ T* s_caller[MV_NC];
    if (t < nb) {
        int arr = 0, c = c0 + t;
        while (c >= a.nc[arr]) c -= a.nc[arr++];
        s_caller[t] = a.ptr[arr] + (int64_t)c * N + k0;
    }
    const int64_t cstep = BLOCKED ? 32 : cs;
    T* const lane_major = lanes + (BLOCKED ? ((int64_t)(l0 >> 5) * L + s0) * (nc * 32) : (int64_t)s0 * NL + l0) + c0 * cstep;
    __syncthreads();
    // f(component of the block, word, place) for all of a side: whole chunks take a
    // place's index for all components, pieces, of one component mostly, are quicker
    // component by component
    auto each = [&](auto side, auto f) {
        if (w == L) {
            side([&](int i, int64_t k) {
#pragma unroll 4
                for (int c = 0; c < nb; ++c) f(c, i, k);
            });
        } else {
            for (int c = 0; c < nb; ++c) side([&](int i, int64_t k) { f(c, i, k); });
        }
    };
    if (TO_LANES) each(caller_side, [&](int c, int i, int64_t k) { copy_async(tiles + c * tile + i, s_caller[c] + k); });
    else each(lane_side, [&](int c, int i, int64_t ix) { copy_async(tiles + c * tile + i, lane_major + c * cstep + ix); });
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (TO_LANES) each(lane_side, [&](int c, int i, int64_t ix) { lane_major[c * cstep + ix] = tiles[c * tile + i]; });
    else each(caller_side, [&](int c, int i, int64_t k) { s_caller[c][k] = tiles[c * tile + i]; });
}

template <typename T>
cudaError_t launch_lanes_move(const LaneArrays<T>& a, T* lanes, int64_t N, int L, int NL, LanesMove how, cudaStream_t st)
{
    constexpr int G = MV_G<T>;
    int nc = 0;
    for (int i = 0; i < a.n; ++i) nc += a.nc[i];
    // as many components a block as its shared memory holds without asking for more
    // (an SM holds four such blocks), fewer where the grid would not fill the SMs
    const int w = std::min(L, MV_W);
    const int64_t pieces = (int64_t)((NL + G - 1) / G) * ((L + MV_W - 1) / MV_W);
    const size_t tile = sizeof(T) * w * mv_row<T>(w);   // at most 33 KB
    const int per_block = (int)std::max<int64_t>(1, std::min<int64_t>({nc, (int64_t)(MV_BYTES / tile), nc * pieces / 608}));
    if (nc > MV_NC) return cudaErrorInvalidValue;
    const size_t smem = tile * per_block;
    const dim3 grid((NL + G - 1) / G, (L + MV_W - 1) / MV_W, (nc + per_block - 1) / per_block);
    auto kern = how == MOVE_OUT  ? lanes_move_kernel<T, false, false>
                : how == MOVE_IN ? lanes_move_kernel<T, true, false>
                                 : lanes_move_kernel<T, true, true>;
    kern<<<grid, MV_THREADS, smem, st>>>(a, lanes, N, L, NL, nc, per_block);
    return cudaGetLastError();
}

template cudaError_t launch_lanes_move<float>(const LaneArrays<float>&, float*, int64_t, int, int, LanesMove, cudaStream_t);
template cudaError_t launch_lanes_move<double>(const LaneArrays<double>&, double*, int64_t, int, int, LanesMove,
                                               cudaStream_t);

// Prior nominal in the lane-major layout: state k of trajectory b gets (m0_b, P0_b).
template <typename T>
__global__ void init_nominal_lanes_kernel(const int64_t* offsets, int B, int64_t N, int L, int NL, const T* m0,
                                          const T* P0, T* x, T* P)
{
    const int64_t cs = (int64_t)L * NL;
    const int64_t total = cs;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int s = (int)(i / NL), l = (int)(i - (int64_t)s * NL);
        const int64_t k = (int64_t)l * L + s;
        if (k >= N) continue;
        const int b = traj_of(offsets, B, k);
        if (x)
#pragma unroll
            for (int c = 0; c < 5; ++c) x[c * cs + i] = m0[5 * b + c];
        if (P)
#pragma unroll
            for (int c = 0; c < 15; ++c) P[c * cs + i] = P0[15 * b + c];
    }
}

template <typename T>
cudaError_t launch_init_nominal_lanes(const int64_t* offsets, int B, int64_t N, int L, int NL, const T* m0,
                                      const T* P0, T* x, T* P, cudaStream_t st)
{
    const int threads = 256;
    const int64_t total = (int64_t)L * NL;
    const int blocks = (int)std::min<int64_t>((total + threads - 1) / threads, 152 * 32);
    init_nominal_lanes_kernel<T><<<blocks, threads, 0, st>>>(offsets, B, N, L, NL, m0, P0, x, P);
    return cudaGetLastError();
}

template cudaError_t launch_init_nominal_lanes<float>(const int64_t*, int, int64_t, int, int, const float*,
                                                      const float*, float*, float*, cudaStream_t);
template cudaError_t launch_init_nominal_lanes<double>(const int64_t*, int, int64_t, int, int, const double*,
                                                       const double*, double*, double*, cudaStream_t);

template <typename T>
__global__ void init_nominal_kernel(const int64_t* offsets, int B, int64_t N, const T* m0, const T* P0, T* x, T* P)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += stride) {
        const int b = traj_of(offsets, B, k);
        if (x)
#pragma unroll
            for (int i = 0; i < 5; ++i) x[i * N + k] = m0[5 * b + i];
        if (P)
#pragma unroll
            for (int i = 0; i < 15; ++i) P[i * N + k] = P0[15 * b + i];
    }
}

template <typename T>
cudaError_t launch_init_nominal(const int64_t* offsets, int B, int64_t N, const T* m0, const T* P0, T* x, T* P,
                                cudaStream_t st)
{
    const int threads = 256;
    const int blocks = (int)std::min<int64_t>((N + threads - 1) / threads, 152 * 32);
    init_nominal_kernel<T><<<blocks, threads, 0, st>>>(offsets, B, N, m0, P0, x, P);
    return cudaGetLastError();
}

// Linearisation in the paper's parametrisation (F, c, Q', H, d, R') of Eq. 11.
template <typename T, int LIN>
__global__ void linearize_kernel(const KParams<T> p, T* F, T* c, T* Qp, T* H, T* d, T* Rp, T* y_used)
{
    if (*(volatile int*)p.status & ST_BADARG) return;
    const int64_t N = p.N;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool ok = true;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += stride) {
        const int b = traj_of(p.offsets, p.B, k);
        const bool has_next = k + 1 < __ldg(p.offsets + b + 1);
        const bool has_obs = k > __ldg(p.offsets + b);
        if (has_next) {
            Trans<T> tr;
            ok &= get_trans<T, LIN>(p, k, tr);
            T Fx[5];
            mv(tr.F, tr.xn, Fx);
#pragma unroll
            for (int i = 0; i < 25; ++i) F[i * N + k] = tr.F[i];
#pragma unroll
            for (int i = 0; i < 5; ++i) c[i * N + k] = tr.fx[i] - Fx[i];
#pragma unroll
            for (int i = 0; i < 15; ++i) Qp[i * N + k] = tr.Q[i];
        } else {
#pragma unroll
            for (int i = 0; i < 25; ++i) F[i * N + k] = T(0);
#pragma unroll
            for (int i = 0; i < 5; ++i) c[i * N + k] = T(0);
#pragma unroll
            for (int i = 0; i < 15; ++i) Qp[i * N + k] = T(0);
        }
        if (has_obs) {
            Obs<T> ob;
            ok &= get_obs<T, LIN>(p, k, b, ob);
            T y[2];
            load_y(p, k, y);
            // h(xn), the measurement y_used and d = zbar - H xn with zbar = y_used - r_offset
            T hx[2];
            if (p.model.kind == MODEL_LINEAR) {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    T v = p.model.d[r];
#pragma unroll
                    for (int l = 0; l < 5; ++l) v = fma(p.model.H[r * 5 + l], ob.xn[l], v);
                    hx[r] = v;
                }
            } else {
                T s[4];
                load_sensors(p.model, b, s);
                bearings(ob.xn, s, hx);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const T yu = (p.model.kind == MODEL_LINEAR) ? y[r] : hx[r] + wrap_angle(y[r] - hx[r]);
                // innovation of x is r - H (x - xn) = yu - (zbar + H (x - xn)), so zbar = yu - r
                T Hx = T(0);
#pragma unroll
                for (int l = 0; l < 5; ++l) Hx = fma(ob.H[r * 5 + l], ob.xn[l], Hx);
                d[r * N + k] = (yu - ob.r[r]) - Hx;
                if (y_used) y_used[r * N + k] = yu;
            }
#pragma unroll
            for (int i = 0; i < 10; ++i) H[i * N + k] = ob.H[i];
#pragma unroll
            for (int i = 0; i < 3; ++i) Rp[i * N + k] = ob.R[i];
        } else {
#pragma unroll
            for (int i = 0; i < 10; ++i) H[i * N + k] = T(0);
#pragma unroll
            for (int i = 0; i < 2; ++i) d[i * N + k] = T(0);
#pragma unroll
            for (int i = 0; i < 3; ++i) Rp[i * N + k] = T(0);
            if (y_used) {
                y_used[k] = T(0);
                y_used[N + k] = T(0);
            }
        }
    }
    if (!ok) atomicOr(p.status, ST_NOT_PD);
}

template <typename T>
cudaError_t launch_linearize(const KParams<T>& p, int lin, T* F, T* c, T* Qp, T* H, T* d, T* Rp, T* y_used,
                             cudaStream_t st)
{
    const int threads = 128;
    const int blocks = (int)std::min<int64_t>((p.N + threads - 1) / threads, 152 * 16);
    if (lin == LIN_IEKS)
        linearize_kernel<T, LIN_IEKS><<<blocks, threads, 0, st>>>(p, F, c, Qp, H, d, Rp, y_used);
    else if (lin == LIN_GH)
        linearize_kernel<T, LIN_GH><<<blocks, threads, 0, st>>>(p, F, c, Qp, H, d, Rp, y_used);
    else
        linearize_kernel<T, LIN_CUBATURE><<<blocks, threads, 0, st>>>(p, F, c, Qp, H, d, Rp, y_used);
    return cudaGetLastError();
}

template cudaError_t launch_init_nominal<float>(const int64_t*, int, int64_t, const float*, const float*, float*,
                                                float*, cudaStream_t);
template cudaError_t launch_init_nominal<double>(const int64_t*, int, int64_t, const double*, const double*,
                                                 double*, double*, cudaStream_t);
template cudaError_t launch_linearize<float>(const KParams<float>&, int, float*, float*, float*, float*, float*,
                                             float*, float*, cudaStream_t);
template cudaError_t launch_linearize<double>(const KParams<double>&, int, double*, double*, double*, double*,
                                              double*, double*, double*, cudaStream_t);

}  // namespace pes
