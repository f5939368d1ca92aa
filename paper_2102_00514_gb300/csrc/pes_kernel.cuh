// The persistent smoother kernel: one cooperative launch runs M iterations of
//   (a) linearisation of every step about the nominal (Eq. 10 or Eqs. 7-9),
//   (b) the forward associative scan of filtering elements (Eqs. 13-15),
//   (c) the reverse associative scan of smoothing elements (Eqs. 17-19),
// and re-linearises about the smoothed means between iterations (Sec. 3).
//
// Scan layout. The N states are split into contiguous chunks of L steps, one per
// thread ("lane"); the first lpb of a block's NT threads are lanes. A lane's filtering element maps the predicted
// state at its chunk's start to the predicted state at the next chunk's start:
// update and predict, step by step. Both scans are three-level
// reduce-then-scans over the lanes:
//   1. every lane folds its chunk into one filtering element;
//   2. a tree over the lane elements of a block in shared memory gives the
//      block's element, published to global memory (pes_tree.cuh);
//   3. after a grid barrier every block reduces the elements of the blocks
//      before it; since the sequence starts with a prior, that is a Gaussian;
//   4. the tree pushes that Gaussian down, so that every lane gets the
//      predicted Gaussian at its chunk's start;
//   5. each lane re-runs its chunk as a Kalman filter from it and keeps the
//      filtered moments.
// The smoothing element of a whole chunk (from the state after it to its first
// state) follows from that Gaussian and the lane's filtering element: the chunk
// is one step of Eq. 17 with the transition (A, b, C) from the state
// conditioned on the chunk's measurements, D = (P^{-1} + J)^{-1}. So the
// smoothing scan needs no fold of per-step elements (350 multiply-adds per
// state), and its levels 2 and 3 do not depend on the filtering re-run: its
// block elements are published before the re-run, which hides the wait for the
// other blocks'. The RTS pass then builds each step's element from the kept
// filtered moments. (Taylor, FP32, T = 2^20: an iteration 245 -> 175 us, of which
// re-run and smoothing up-sweep 100 -> 40, the wait for the smoothing elements 16
// -> 1, RTS 35 -> 50.)
//
// What bounds it at that size: the sequential passes (fold 34, re-run 32, RTS 50
// us) are issue-bound with two warps per sub-partition at 255 registers, the
// trees (34 + 16 us) are levels of one operator's latency.
//
// In FP32, within a chunk means are kept as deviations from the nominal (the
// filter's, the fold's and the smoother's), re-referenced from state to state by
// the difference of their nominals, and the trees' elements carry reference points: positions of
// tens to thousands of units would otherwise be rounded at every step and level,
// and the rounding of the means is what the next iteration's linearisation
// amplifies (batch of 1,024 trajectories after three FP32 iterations, against 64
// bits: means 6.1e-7 -> 1.0e-7, covariances 7e-6 -> 2.5e-6).
//
// A chunk's passes read only its own states' nominal, so no barrier separates
// iterations: the block aggregates are double-buffered, and a block can reach
// the aggregates of iteration i + 2 only after every block has passed the first
// barrier of iteration i + 1, that is, has read those of iteration i. Only the
// tolerance mode waits for all blocks at an iteration's end.
//
// Grid barriers spin on a global counter with a wall-clock limit; on timeout
// they set ST_TIMEOUT and return, so the kernel always terminates.
#pragma once

#include "pes_async.cuh"
#include "pes_tree.cuh"

namespace pes {

enum { MODE_FILTER = 0, MODE_SMOOTH = 1, MODE_RUN = 2 };

constexpr int HAND = 20;          // filtered moments kept per state
constexpr int LINS = 65;          // stored linearisation scalars per state, at most

// The compiled forms of the smoother: the linearisation, and whether the model
// is known to be the coordinated turn (the structure of its slopes, and no code
// for the linear model in the loops) or is looked up (_ANY); the scans over given
// arrays read lane-major copies of them or the arrays themselves (_IN_PLACE).
enum { KK_ARRAYS = 0, KK_IEKS = 1, KK_CUBATURE = 2, KK_GH = 3, KK_IEKS_ANY = 4, KK_CUBATURE_ANY = 5, KK_ARRAYS_IN_PLACE = 6 };
template <int K>
constexpr int kLinOf = K == KK_IEKS_ANY ? LIN_IEKS
                       : K == KK_CUBATURE_ANY ? LIN_CUBATURE
                       : K == KK_ARRAYS_IN_PLACE ? LIN_ARRAYS : K;
template <int K>
constexpr bool kArrays = kLinOf<K> == LIN_ARRAYS;
template <int K>
constexpr int kFS = K == KK_IEKS ? FS_CT : (K == KK_CUBATURE ? FS_SLR : FS_DENSE);

// Whether the fold hands its linearisation of every state to the later passes
// instead of their linearising again. The sigma-point linearisations cost far
// more than the traffic; the Taylor one does not.
template <int K>
constexpr bool kStoreLin = kSigma<kLinOf<K>>;
// Scalars stored per state; the transition's are kLinTrans of them, from
// kLinTransAt. Compact form (the coordinated turn's cubature regression): F rows
// 0-3 (20), fx (4; less xn in FP32), Q' (10), H (4), r (2), R' (3); the nominal is read
// from the trajectory, the rest is constant. Dense form: H (10), r (2), R' (3),
// xn (5), F (25), fx (5), Q' (15).
template <int K>
constexpr int kLinScalars = K == KK_CUBATURE ? 43 : LINS;
template <int K>
constexpr int kLinTransAt = K == KK_CUBATURE ? 0 : 15;
template <int K>
constexpr int kLinTrans = K == KK_CUBATURE ? 34 : 50;
// Stream stages: of the re-run (beside the smoother's tree, which is live), and
// of the RTS pass.
template <int K>
constexpr int kLinStages = K == KK_CUBATURE ? 2 : 1;
template <int K>
constexpr int kRtsStages = (kStoreLin<K> && K != KK_CUBATURE) ? 3 : 4;
constexpr int kMaxStages = 4;
// Whether the trees keep combine_filter's rounding (fold_filter_arrays).
template <int K, typename T>
constexpr bool kKeepRounding = kArrays<K> && sizeof(T) == 4;

template <typename T>
struct KParams {
    int64_t N;
    const int64_t* offsets;   // [B+1], device
    int B;
    int mode;
    int iters;                // RUN: maximum iterations; otherwise 1
    double tol;               // RUN: relative update-norm tolerance (<= 0: fixed iterations)
    int write_P_every_iter;   // RUN: write smoothed covariances in every iteration
    DevModel<T> model;
    // per-state arrays, component-major with stride cs. In the scans they are in
    // the kernel's lane-major layout; the element-wise kernels and the sequential
    // smoother use the caller's (cs = N).
    const T* y;               // [2] (slot of each x_0 ignored)
    const T* m0;              // [B][5]
    const T* P0;              // [B][15]
    // filtered moments (MODE_FILTER output)
    T* xf;
    T* Pf;
    // smoothed moments: MODE_SMOOTH output; MODE_RUN nominal (in place) and output
    T* x;
    T* P;
    // workspace
    T* hand;           // MODE_RUN: filtered moments, kept for the RTS pass: [warp][s][HAND][32 lanes]
    // MODE_RUN: the sigma-point linearisation, handed from the fold to the later
    // passes; MODE_FILTER / MODE_SMOOTH: the given arrays' copy: [warp][s][component][32]
    T* lin;
    // MODE_FILTER / MODE_SMOOTH, in_place (KK_ARRAYS_IN_PLACE): the given arrays
    // themselves, [component][N], results in the caller's arrays too (cs = N)
    const T* arr[7];   // F, c, Q', H, d, R', y or F, c, Q', filtered mean and covariance
    int in_place;
    T* aggF;           // [2][agg_blocks][FE]: the blocks' filtering elements, by iteration parity
    T* aggS;           // [2][agg_blocks][SE]: their smoothing elements
    int agg_blocks;    // blocks the aggregates have room for
    unsigned* bar;     // grid barrier counter, zero at launch
    int* status;       // ST_* bits
    double* conv;      // [2][B][2] update-norm accumulators, zero at launch
    int* iters_done;
    int* traj_iters;   // RUN with tol > 0: [B], the first iteration whose update met tol (0: none); or NULL
    double* loglik;    // FILTER: [B] log p(y_{1:T_b}) accumulated (zero at launch), or NULL
    int L;             // steps per lane
    int lpb;           // lanes per block: a multiple of 32, at most NT
    int NL;            // lanes = NB * lpb
    int64_t cs;        // component stride of the per-state arrays
    long long timeout_ns;
    long long* ptime;  // optional per-block phase timestamps of the first iteration (NULL: off)
};

constexpr int NPHASE = 16;
// Phase timestamps: thread 0 of every block records %globaltimer at the phase
// boundaries of the first iteration when p.ptime is set.
#define PES_PHASE(p, it, i)                                                        \
    do {                                                                           \
        if ((p).ptime && (it) == 0 && threadIdx.x == 0)                            \
            (p).ptime[(size_t)blockIdx.x * NPHASE + (i)] = globaltimer_ns();      \
    } while (0)

// ---- small device utilities ------------------------------------------------

PES_DEV long long globaltimer_ns()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

PES_DEV unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid-wide barrier for a cooperative launch (all blocks co-resident), in two
// halves: arrive publishes the block's earlier writes, wait returns once every
// block has arrived.
template <typename T>
PES_DEV void grid_arrive(const KParams<T>& p, unsigned& gen)
{
    __syncthreads();
    ++gen;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(p.bar, 1u);
    }
}

template <typename T>
PES_DEV void grid_wait(const KParams<T>& p, unsigned gen)
{
    if (threadIdx.x == 0) {
        const unsigned target = gen * gridDim.x;
        const long long t0 = globaltimer_ns();
        unsigned polls = 0;
        while (ld_acquire(p.bar) < target) {
            if (*(volatile int*)p.status & ST_TIMEOUT) break;
            if (++polls > (1u << 26) || globaltimer_ns() - t0 > p.timeout_ns) {
                atomicOr(p.status, ST_TIMEOUT);
                break;
            }
            __nanosleep(32);
        }
        __threadfence();
    }
    __syncthreads();
}

// Trajectory cursor over the CSR offsets.
struct SegCursor {
    const int64_t* off;
    int b;
    int64_t head, next;
    PES_DEV void init(const int64_t* o, int B, int64_t k)
    {
        off = o;
        int lo = 0, hi = B - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(o + mid) <= k) lo = mid;
            else hi = mid - 1;
        }
        b = lo;
        head = __ldg(o + b);
        next = __ldg(o + b + 1);
    }
    PES_DEV void forward(int64_t k)
    {
        while (k >= next) {
            ++b;
            head = next;
            next = __ldg(off + b + 1);
        }
    }
    PES_DEV void backward(int64_t k)
    {
        while (k < head) {
            --b;
            next = head;
            head = __ldg(off + b);
        }
    }
    PES_DEV bool is_head(int64_t k) const { return k == head; }
    PES_DEV bool is_tail(int64_t k) const { return k == next - 1; }
};

template <typename T>
PES_DEV void load_prior(const KParams<T>& p, int b, T* m0, T* P0)
{
#pragma unroll
    for (int i = 0; i < 5; ++i) m0[i] = __ldg(p.m0 + 5 * b + i);
#pragma unroll
    for (int i = 0; i < 15; ++i) P0[i] = __ldg(p.P0 + 15 * b + i);
}

// The nominal trajectory is rewritten by every iteration. A lane reads only its own
// states' nominal, which it wrote itself in the iteration before (the first one finds
// an earlier kernel's), so plain loads need no barrier between iterations; they are
// L1-cached, and consecutive steps of a warp's lanes share cache sectors.
template <typename T>
PES_DEV void load_nominal(const KParams<T>& p, int64_t ix, T* x)
{
#pragma unroll
    for (int i = 0; i < 5; ++i) x[i] = p.x[i * p.cs + ix];
}

template <typename T>
PES_DEV void load_nominal_cov(const KParams<T>& p, int64_t ix, T* P)
{
#pragma unroll
    for (int i = 0; i < 15; ++i) P[i] = p.P[i * p.cs + ix];
}

template <typename T>
PES_DEV void load_y(const KParams<T>& p, int64_t ix, T* y)
{
    y[0] = __ldg(p.y + ix);
    y[1] = __ldg(p.y + p.cs + ix);
}

// Place of step s of a lane in the per-state arrays: [component][step][lane], in
// which a warp's accesses at one step are contiguous.
template <typename T>
PES_DEV int64_t lane_ix(const KParams<T>& p, int64_t s, int lane)
{
    return s * p.NL + lane;
}

// ---- linearisation of one step ------------------------------------------------

// Per-state inputs of the linearisation, loaded one step ahead of their use
// so that the loads overlap the previous step's arithmetic.
template <typename T, int LIN>
struct StateIn {
    T x[5];    // nominal mean (IEKS, cubature)
    T P[15];   // nominal covariance (cubature)
    T y[2];    // measurement
};

template <typename T, int LIN>
PES_DEV void load_state(const KParams<T>& p, int64_t ix, StateIn<T, LIN>& s)
{
    load_nominal(p, ix, s.x);
    if (kSigma<LIN>) load_nominal_cov(p, ix, s.P);
    load_y(p, ix, s.y);
}

// Sigma-point factor of the state's nominal covariance (cubature only).
template <typename T, int LIN>
struct Factor {
    T L[kSigma<LIN> ? 25 : 1];
    T rd[kSigma<LIN> ? 5 : 1];
};

template <typename T, int LIN>
PES_DEV bool factor_state(const StateIn<T, LIN>& s, Factor<T, LIN>& f)
{
    if (kSigma<LIN>) return cub_factor(s.P, f.L, f.rd);
    return true;
}

// Transition k -> k+1 (Eq. 10 or Eq. 7).
template <typename T, int LIN>
PES_DEV void lin_trans(const KParams<T>& p, const StateIn<T, LIN>& s, const Factor<T, LIN>& f, Trans<T>& tr)
{
    if (LIN == LIN_IEKS) lin_trans_taylor(p.model, s.x, tr);
    else if (LIN == LIN_GH) lin_trans_gh(p.model, s.x, f.L, f.rd, tr);
    else lin_trans_cubature(p.model, s.x, f.L, f.rd, tr);
}

// Observation at k (Eq. 10 or Eq. 9).
template <typename T, int LIN>
PES_DEV void lin_obs(const KParams<T>& p, int b, const StateIn<T, LIN>& s, const Factor<T, LIN>& f, Obs<T>& ob)
{
    if (LIN == LIN_IEKS) lin_obs_taylor(p.model, b, s.x, s.y, ob);
    else if (LIN == LIN_GH) lin_obs_gh(p.model, b, s.x, f.L, f.rd, s.y, ob);
    else lin_obs_cubature(p.model, b, s.x, f.L, f.rd, s.y, ob);
}

// One-shot forms used by the stand-alone linearisation kernel.
template <typename T, int LIN>
PES_DEV bool get_trans(const KParams<T>& p, int64_t ix, Trans<T>& tr)
{
    StateIn<T, LIN> s;
    load_state(p, ix, s);
    Factor<T, LIN> f;
    const bool ok = factor_state(s, f);
    lin_trans(p, s, f, tr);
    return ok;
}

template <typename T, int LIN>
PES_DEV bool get_obs(const KParams<T>& p, int64_t ix, int b, Obs<T>& ob)
{
    StateIn<T, LIN> s;
    load_state(p, ix, s);
    Factor<T, LIN> f;
    const bool ok = factor_state(s, f);
    lin_obs(p, b, s, f, ob);
    return ok;
}

// The linearisation of a compiled form of the smoother; fx is f(xn) - xn where kRel.
template <int K, typename T>
PES_DEV void form_trans(const KParams<T>& p, const StateIn<T, kLinOf<K>>& s, const Factor<T, kLinOf<K>>& f,
                        Trans<T>& tr)
{
    if constexpr (K == KK_IEKS) ct_trans_taylor(p.model, s.x, tr);
    else if constexpr (K == KK_CUBATURE) ct_trans_cubature(p.model, s.x, f.L, f.rd, tr);
    else {
        lin_trans<T, kLinOf<K>>(p, s, f, tr);
#pragma unroll
        for (int i = 0; i < 5 && kRel<T>; ++i) tr.fx[i] -= tr.xn[i];
    }
}

template <int K, typename T>
PES_DEV void form_obs(const KParams<T>& p, int b, const StateIn<T, kLinOf<K>>& s,
                      const Factor<T, kLinOf<K>>& f, Obs<T>& ob)
{
    if constexpr (K == KK_IEKS) ct_obs_taylor(p.model, b, s.x, s.y, ob);
    else if constexpr (K == KK_CUBATURE) ct_obs_cubature(p.model, b, s.x, f.L, f.rd, s.y, ob);
    else lin_obs<T, kLinOf<K>>(p, b, s, f, ob);
}

// ---- lane-level passes -------------------------------------------------------------

// Stored linearisation, [warp][s][kLinScalars][32 lanes].
template <int K, typename T>
PES_DEV T* lin_slot(const KParams<T>& p, int s, int lane)
{
    return p.lin + ((size_t)(lane >> 5) * p.L + s) * (kLinScalars<K> * 32) + (lane & 31);
}

template <int K, typename T>
PES_DEV void store_lin_obs(const KParams<T>& p, int s, int lane, const Obs<T>& ob)
{
    T* h = lin_slot<K>(p, s, lane);
    if constexpr (K == KK_CUBATURE) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            h[(34 + 2 * r) * 32] = ob.H[r * 5];
            h[(35 + 2 * r) * 32] = ob.H[r * 5 + 1];
            h[(38 + r) * 32] = ob.r[r];
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) h[(40 + i) * 32] = ob.R[i];
    } else {
#pragma unroll
        for (int i = 0; i < 5; ++i) h[(15 + i) * 32] = ob.xn[i];
#pragma unroll
        for (int i = 0; i < 10; ++i) h[i * 32] = ob.H[i];
        h[10 * 32] = ob.r[0];
        h[11 * 32] = ob.r[1];
#pragma unroll
        for (int i = 0; i < 3; ++i) h[(12 + i) * 32] = ob.R[i];
    }
}

// packed index of entry q of the leading 4x4 block of a symmetric 5x5 matrix
__host__ __device__ constexpr int si4(int q) { return q < 4 ? q : (q < 7 ? q + 1 : (q < 9 ? q + 2 : q + 3)); }

template <int K, typename T>
PES_DEV void store_lin_trans(const KParams<T>& p, int s, int lane, const Trans<T>& tr)
{
    T* h = lin_slot<K>(p, s, lane);
    if constexpr (K == KK_CUBATURE) {
#pragma unroll
        for (int i = 0; i < 20; ++i) h[i * 32] = tr.F[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) h[(20 + i) * 32] = tr.fx[i];
#pragma unroll
        for (int i = 0; i < 10; ++i) h[(24 + i) * 32] = tr.Q[si4(i)];
    } else {
#pragma unroll
        for (int i = 0; i < 5; ++i) h[(15 + i) * 32] = tr.xn[i];
#pragma unroll
        for (int i = 0; i < 25; ++i) h[(20 + i) * 32] = tr.F[i];
#pragma unroll
        for (int i = 0; i < 5; ++i) h[(45 + i) * 32] = tr.fx[i];
#pragma unroll
        for (int i = 0; i < 15; ++i) h[(50 + i) * 32] = tr.Q[i];
    }
}

// The slot range of a lane's warp at step s.
template <int K, typename T>
PES_DEV const T* lin_warp(const KParams<T>& p, int s, int lane)
{
    return p.lin + ((size_t)(lane >> 5) * p.L + s) * (kLinScalars<K> * 32);
}

// Per-thread asynchronous prefetch of the next states' inputs into shared
// memory: NS components of a state, consecutive rows of the per-state arrays from
// `src` on. For the sigma-point folds, whose register pressure rules out a
// register prefetch (nominal mean and covariance, measurement). Each thread
// copies its own scalars with cp.async and reads only its own stages back, so no
// block synchronisation is involved. Element c of stage i sits at base[(i * NS + c) * stride] (thread-contiguous columns).
template <typename T, int NS>
struct Prefetch {
    T* base;
    int stride;
    const T* src;
    int64_t cs;
    PES_DEV void issue(int64_t ix, int i) const
    {
        T* d = base + (size_t)i * NS * stride;
        const T* q = src + ix;
#pragma unroll
        for (int c = 0; c < NS; ++c)
            asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(d + c * stride)), "l"(q + c * cs),
                         "n"(sizeof(T))
                         : "memory");
    }
    PES_DEV static void commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
    // all but the most recent group complete
    PES_DEV static void wait_prev() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
    PES_DEV static void wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
    PES_DEV T get(int i, int c) const { return base[((size_t)i * NS + c) * stride]; }
};
constexpr int kStateIn = 22;    // a run's inputs: x, P, y
// The scans over given arrays stream a state's components: the filter's F, c, Q',
// H, d, R', y (three stages in the re-run, where a step needs the one before it
// too), the smoother's F, c, Q' and filtered mean and covariance.
constexpr int kFilterIn = 62, kSmoothIn = 65;
template <typename T>
using FoldStream = WarpStream<T, kFilterIn, 2>;
template <typename T>
using FilterStream = WarpStream<T, kFilterIn, 3>;
template <typename T>
using SmoothStream = WarpStream<T, kSmoothIn, 2>;
// The slot range of a lane's warp at step s, [warp][s][NC][32 lanes].
template <int NC, typename T>
PES_DEV const T* array_warp(const KParams<T>& p, int s, int lane)
{
    return p.lin + ((size_t)(lane >> 5) * p.L + s) * (NC * 32);
}

// The same components of state k from the caller's arrays, NC of them in all.
template <typename T, int NC>
struct ArrayState {
    const KParams<T>& p;
    int64_t k;
    // (read-only loads: the results' arrays may be the filtered moments', but a lane
    // reads a state before it writes it, and no other lane reads it)
    PES_DEV T at(int arr, int c) const { return __ldg(p.arr[arr] + c * p.N + k); }
    PES_DEV T get(int, int c) const
    {
        if (c < 25) return at(0, c);
        if (c < 30) return at(1, c - 25);
        if (c < 45) return at(2, c - 30);
        if (NC == kSmoothIn) return c < 50 ? at(3, c - 45) : at(4, c - 50);
        if (c < 55) return at(3, c - 45);
        if (c < 57) return at(4, c - 55);
        return c < 60 ? at(5, c - 57) : at(6, c - 60);
    }
};

// Place of state k = a + s of a lane in the scans' outputs.
template <bool IP, typename T>
PES_DEV int64_t array_ix(const KParams<T>& p, int64_t k, int s, int lane)
{
    return IP ? k : lane_ix(p, s, lane);
}

template <typename T, class S>
PES_DEV void array_trans(const S& q, int i, Trans<T>& tr)
{
#pragma unroll
    for (int c = 0; c < 25; ++c) tr.F[c] = q.get(i, c);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
        tr.fx[c] = q.get(i, 25 + c);
        tr.xn[c] = T(0);
    }
#pragma unroll
    for (int c = 0; c < 15; ++c) tr.Q[c] = q.get(i, 30 + c);
}

template <typename T, class S>
PES_DEV void array_obs(const S& q, int i, Obs<T>& ob)
{
#pragma unroll
    for (int c = 0; c < 10; ++c) ob.H[c] = q.get(i, 45 + c);
#pragma unroll
    for (int r = 0; r < 2; ++r) ob.r[r] = q.get(i, 60 + r) - q.get(i, 55 + r);
#pragma unroll
    for (int c = 0; c < 3; ++c) ob.R[c] = q.get(i, 57 + c);
#pragma unroll
    for (int c = 0; c < 5; ++c) ob.xn[c] = T(0);
}

// The transition out of state a - 1, the last one of the lane before `lane`.
template <bool IP, typename T>
PES_DEV void load_array_trans(const KParams<T>& p, int64_t a, int lane, Trans<T>& tr)
{
    if constexpr (IP) {
        array_trans(ArrayState<T, kFilterIn>{p, a - 1}, 0, tr);
        return;
    }
    const T* h = array_warp<kFilterIn>(p, p.L - 1, lane - 1) + ((lane - 1) & 31);
#pragma unroll
    for (int i = 0; i < 25; ++i) tr.F[i] = __ldg(h + i * 32);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        tr.fx[i] = __ldg(h + (25 + i) * 32);
        tr.xn[i] = T(0);
    }
#pragma unroll
    for (int i = 0; i < 15; ++i) tr.Q[i] = __ldg(h + (30 + i) * 32);
}

// acc <- acc (x) the Levenberg-Marquardt pseudo-measurement of a state's nominal
// xb (the zero deviation where kRel). Out of line: a damped run pays for the call,
// the others keep the operator's code and registers out of their loops.
template <typename T>
__device__ __noinline__ void damp_element(FElem<T>& acc, const T* xb, T lambda)
{
    FElem<T> dmp;
    felem_damping(dmp, xb, lambda);
    combine_filter(acc, dmp, acc);
}

template <typename T>
__device__ __noinline__ void damp_gauss(Gauss<T>& g, const T* xb, T lambda)
{
    FElem<T> dmp;
    felem_damping(dmp, xb, lambda);
    apply_filter(g, dmp, g);
}

// Filtering, level 1: fold the lane's chunk [a, e) into one element, from the
// predicted state at a to the predicted state at e. Step k folds the update
// with its own observation and then the prediction through its outgoing
// transition (k -> k+1), both linearised about the nominal of k, so the state's
// sigma-point factor serves both. With a stored linearisation (MODE_RUN,
// sigma-point rules) both are kept for the re-run and the RTS pass.
template <int K, typename T>
PES_DEV bool fold_filter_chunk(const KParams<T>& p, int64_t a, int64_t e, int lane, FElem<T>& acc,
                               const Prefetch<T, kStateIn>& pf)
{
    constexpr int LIN = kLinOf<K>, FS = kFS<K>;
    bool ok = true;
    T zero[5] = {T(0), T(0), T(0), T(0), T(0)};
    felem_identity(acc, zero);
    if (a >= e) return ok;
    const bool store_lin = kStoreLin<K> && p.mode == MODE_RUN;
    SegCursor cur;
    cur.init(p.offsets, p.B, a);
    const int64_t dix = p.NL;
    int64_t ix = lane;
    StateIn<T, LIN> sc, sn;   // inputs of states k, k+1
    // the next state's inputs are loaded a step ahead: into registers for
    // the Taylor linearisation; for the sigma-point ones, whose register
    // pressure makes a register prefetch cost more in spills than it hides,
    // into shared memory, three stages: the state before is still needed
    int st = 0;
    constexpr bool prefetch = !kSigma<LIN>;
    if (prefetch) {
        load_state(p, ix, sc);
    } else {
        pf.issue(ix, 0);
        pf.commit();
    }
#pragma unroll 1
    for (int64_t k = a;; ++k, ix += dix) {
        cur.forward(k);
        const int s = (int)(k - a);
        if (prefetch) {
            if (k + 1 < e) load_state(p, ix + dix, sn);
        } else {
            if (k + 1 < e) pf.issue(ix + dix, st == 2 ? 0 : st + 1);
            pf.commit();
            pf.wait_prev();
#pragma unroll
            for (int i = 0; i < 5; ++i) sc.x[i] = pf.get(st, i);
#pragma unroll
            for (int i = 0; i < 15; ++i) sc.P[i] = pf.get(st, 5 + i);
            sc.y[0] = pf.get(st, 20);
            sc.y[1] = pf.get(st, 21);
        }
        if (!kRel<T> && s == 0) {   // the input is measured from the nominal of a
            felem_identity(acc, sc.x);
        } else if (kRel<T> && !prefetch && s > 0) {
#pragma unroll
            for (int i = 0; i < 5; ++i) acc.b[i] += pf.get(st == 0 ? 2 : st - 1, i) - sc.x[i];
        }
        Factor<T, LIN> fc;
        ok &= factor_state(sc, fc);
        if (cur.is_head(k)) {
            T m0[5], P0[15];
            load_prior(p, cur.b, m0, P0);
#pragma unroll
            for (int i = 0; i < 5 && kRel<T>; ++i) m0[i] -= sc.x[i];
            felem_apply_prior(acc, m0, P0);
        } else {
            Obs<T> ob;
            form_obs<K>(p, cur.b, sc, fc, ob);
            if (store_lin) store_lin_obs<K>(p, s, lane, ob);
            ok &= fold_update<FS, kRel<T>>(acc, ob);
        }
        if (lm_of(p.model, cur.b) > T(0)) {
            FElem<T> tmp = acc;
            T xb[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) xb[i] = kRel<T> ? T(0) : sc.x[i];
            damp_element(tmp, xb, lm_of(p.model, cur.b));
            acc = tmp;
        }
        if (!cur.is_tail(k)) {
            Trans<T> tr;
            form_trans<K>(p, sc, fc, tr);
            if (store_lin) store_lin_trans<K>(p, s, lane, tr);
            fold_predict<FS, kRel<T>>(acc, tr);
        }
        if (k + 1 == e) break;
        // from the next state's nominal on
        if (prefetch) {
#pragma unroll
            for (int i = 0; i < 5 && kRel<T>; ++i) acc.b[i] += sc.x[i] - sn.x[i];
            sc = sn;
        }
        st = st == 2 ? 0 : st + 1;
    }
    // the reference points: of the output the last nominal, of the input the first
    // (read again, which takes the loop fewer registers than keeping it)
    if (kRel<T>) {
        felem_set_ref(acc, sc.x);
        load_nominal(p, lane, acc.xr);
    }
    if (!prefetch) pf.wait_all();
    if (store_lin) stores_before_bulk_reads();   // the re-run and the RTS pass stream them, after block barriers
    return ok;
}

// The same over given arrays (the filter scan). Its chunks' boundaries are the
// filtered states, each step predicting from the previous state and then
// updating: its results keep the rounding that they always had, which the FP64
// log-likelihoods of FP32 runs show. IP: from the caller's arrays in place, without
// a stream.
template <bool IP, typename T>
PES_DEV bool fold_filter_arrays(const KParams<T>& p, int64_t a, int64_t e, int lane, int steps, FElem<T>& acc, T* wstage,
                                uint64_t* wbar, uint32_t& wpar)
{
    bool ok = true;
    T zero[5] = {T(0), T(0), T(0), T(0), T(0)};
    felem_identity(acc, zero);
    FoldStream<T> ws;
    ws.init(wstage, wbar, wpar);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        if (!IP && i < steps) ws.issue(array_warp<kFilterIn>(p, i, lane), i);
    SegCursor cur;
    if (a < e) {
        cur.init(p.offsets, p.B, a);
        if (!cur.is_head(a)) {   // the transition out of the previous lane's last state
            Trans<T> tr;
            load_array_trans<IP>(p, a, lane, tr);
            fold_predict(acc, tr);
        }
    }
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
        const int64_t k = a + s;
        const int st = s & 1;
        const ArrayState<T, kFilterIn> own{p, k};
        if (!IP) ws.wait(st, p.status);
        if (k < e) {
            cur.forward(k);
            if (cur.is_head(k)) {
                T m0[5], P0[15];
                load_prior(p, cur.b, m0, P0);
                felem_apply_prior(acc, m0, P0);
            } else {
                Obs<T> ob;
                if constexpr (IP) array_obs(own, 0, ob);
                else array_obs(ws, st, ob);
                ok &= fold_update(acc, ob);
            }
            if (!cur.is_tail(k) && k + 1 < e) {
                Trans<T> tr;
                if constexpr (IP) array_trans(own, 0, tr);
                else array_trans(ws, st, tr);
                fold_predict(acc, tr);
            }
        }
        if (IP) continue;
        __syncwarp();
        if (s + 2 < steps) ws.issue(array_warp<kFilterIn>(p, s + 2, lane), st);
    }
    if (!IP) wpar = ws.parity;
    return ok;
}

// Filtered moments in the given arrays (MODE_FILTER output).
template <typename T>
PES_DEV void store_filtered(const KParams<T>& p, int64_t ix, const T* m, const T* P)
{
#pragma unroll
    for (int i = 0; i < 5; ++i) p.xf[i * p.cs + ix] = m[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) p.Pf[i * p.cs + ix] = P[i];
}

// MODE_RUN: the filtered moments (x*, in FP32 less the nominal, P*) of state a + s of a lane, kept
// between the filtering re-run and the RTS pass, which builds the smoothing
// element from them (20 scalars per state; handing over finished elements, 50
// scalars, cost more in traffic than the element's prediction does in
// arithmetic). Layout [warp][s][component][32 lanes]: a warp's accesses for one
// step are one contiguous, coalesced run.
template <typename T>
PES_DEV void store_xP(const KParams<T>& p, int s, int lane, const T* m, const T* P)
{
    T* h = p.hand + ((size_t)(lane >> 5) * p.L + s) * (HAND * 32) + (lane & 31);
#pragma unroll
    for (int i = 0; i < 5; ++i) h[i * 32] = m[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) h[(5 + i) * 32] = P[i];
}

// The linearisation of stage `i` of a stream (layout of store_lin_*; `off` is
// what precedes slot component 0 in the stage); xn the state's nominal (read
// where it is not stored).
template <int K, typename T, class S>
PES_DEV void obs_from_stage(const S& ws, int i, const T* xn, Obs<T>& ob)
{
    if constexpr (K == KK_CUBATURE) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            ob.H[r * 5] = ws.get(i, 34 + 2 * r);
            ob.H[r * 5 + 1] = ws.get(i, 35 + 2 * r);
            ob.r[r] = ws.get(i, 38 + r);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) ob.R[c] = ws.get(i, 40 + c);
#pragma unroll
        for (int c = 0; c < 5; ++c) ob.xn[c] = xn[c];
    } else {
#pragma unroll
        for (int c = 0; c < 10; ++c) ob.H[c] = ws.get(i, c);
        ob.r[0] = ws.get(i, 10);
        ob.r[1] = ws.get(i, 11);
#pragma unroll
        for (int c = 0; c < 3; ++c) ob.R[c] = ws.get(i, 12 + c);
#pragma unroll
        for (int c = 0; c < 5; ++c) ob.xn[c] = ws.get(i, 15 + c);
    }
}

template <int K, typename T, class S>
PES_DEV void trans_from_stage(const KParams<T>& p, const S& ws, int i, int off, const T* xn, Trans<T>& tr)
{
    if constexpr (K == KK_CUBATURE) {
#pragma unroll
        for (int c = 0; c < 20; ++c) tr.F[c] = ws.get(i, off + c);
#pragma unroll
        for (int c = 0; c < 4; ++c) tr.fx[c] = ws.get(i, off + 20 + c);
        tr.fx[4] = kRel<T> ? T(0) : xn[4];
#pragma unroll
        for (int c = 0; c < 15; ++c) tr.Q[c] = p.model.Q[c];
#pragma unroll
        for (int c = 0; c < 10; ++c) tr.Q[si4(c)] = ws.get(i, off + 24 + c);
#pragma unroll
        for (int c = 0; c < 5; ++c) tr.xn[c] = xn[c];
    } else {
#pragma unroll
        for (int c = 0; c < 5; ++c) tr.xn[c] = ws.get(i, off + 15 + c);
#pragma unroll
        for (int c = 0; c < 25; ++c) tr.F[c] = ws.get(i, off + 20 + c);
#pragma unroll
        for (int c = 0; c < 5; ++c) tr.fx[c] = ws.get(i, off + 45 + c);
#pragma unroll
        for (int c = 0; c < 15; ++c) tr.Q[c] = ws.get(i, off + 50 + c);
    }
}

// Filtering, level 5: re-run the chunk from the predicted Gaussian at its start,
// keeping the filtered moments. The loop runs over the L steps of the chunk in
// every lane of the warp (lanes whose chunk is shorter idle), so that a warp
// stream can feed it the stored linearisation.
template <int K, typename T>
PES_DEV bool rerun_filter_chunk(const KParams<T>& p, int64_t a, int64_t e, int lane, int steps, const Gauss<T>& G, T* wstage,
                                uint64_t* wbar, uint32_t& wpar)
{
    constexpr int LIN = kLinOf<K>, FS = kFS<K>, ST = kLinStages<K>;
    bool ok = true;
    const bool any = a < e;
    constexpr bool use_lin = kStoreLin<K>;
    SegCursor cur;
    if (any) cur.init(p.offsets, p.B, a);
    T m[5], P[15];
#pragma unroll
    for (int i = 0; i < 5; ++i) m[i] = G.m[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) P[i] = G.P[i];
    const int64_t dix = p.NL;
    int64_t ix = lane;
    StateIn<T, LIN> sc, sn;   // inputs of states k, k+1 (when linearising here)
    T xc[5], xn[5];   // nominals of states k, k+1
    if (any) {
        if (use_lin) load_nominal(p, ix, xc);
        else load_state(p, ix, sc);
    }
    WarpStream<T, kLinScalars<K>, ST> ws;
    if (use_lin) {
        ws.init(wstage, wbar, wpar);
#pragma unroll
        for (int i = 0; i < ST; ++i)
            if (i < steps) ws.issue(lin_warp<K>(p, i, lane), i);
    }
#pragma unroll 1
    for (int s = 0; s < steps; ++s, ix += dix) {
        const int64_t k = a + s;
        const int st = s % ST;
        if (use_lin) ws.wait(st, p.status);
        if (k < e) {
            cur.forward(k);
            if (!use_lin && k + 1 < e) load_state(p, ix + dix, sn);
            if (use_lin && k + 1 < e) load_nominal(p, ix + dix, xn);
            Factor<T, LIN> fc;
            if (!use_lin) ok &= factor_state(sc, fc);
            if (!use_lin)
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    xc[i] = sc.x[i];
                    xn[i] = sn.x[i];
                }
            if (kRel<T> && s == 0)
#pragma unroll
                for (int i = 0; i < 5; ++i) m[i] += G.r[i] - xc[i];
            if (cur.is_head(k)) {
                load_prior(p, cur.b, m, P);
#pragma unroll
                for (int i = 0; i < 5 && kRel<T>; ++i) m[i] -= xc[i];
            } else {
                Obs<T> ob;
                if constexpr (use_lin) obs_from_stage<K>(ws, st, xc, ob);
                else form_obs<K>(p, cur.b, sc, fc, ob);
                T mn[5], Pn[15];
                ok &= kf_update<FS, kRel<T>>(ob, m, P, mn, Pn);
#pragma unroll
                for (int i = 0; i < 5; ++i) m[i] = mn[i];
#pragma unroll
                for (int i = 0; i < 15; ++i) P[i] = Pn[i];
            }
            if (lm_of(p.model, cur.b) > T(0)) {
                Gauss<T> g;
#pragma unroll
                for (int i = 0; i < 5; ++i) g.m[i] = m[i];
#pragma unroll
                for (int i = 0; i < 15; ++i) g.P[i] = P[i];
                T xb[5];
#pragma unroll
                for (int i = 0; i < 5; ++i) xb[i] = kRel<T> ? T(0) : xc[i];
                damp_gauss(g, xb, lm_of(p.model, cur.b));
#pragma unroll
                for (int i = 0; i < 5; ++i) m[i] = g.m[i];
#pragma unroll
                for (int i = 0; i < 15; ++i) P[i] = g.P[i];
            }
            store_xP(p, s, lane, m, P);
            if (k + 1 < e && !cur.is_tail(k)) {
                Trans<T> tr;
                if constexpr (use_lin) trans_from_stage<K>(p, ws, st, 0, xc, tr);
                else form_trans<K>(p, sc, fc, tr);
                T mp[5], FP[25], Pp[15];
                predict<FS, kRel<T>>(tr, m, P, mp, FP, Pp);
#pragma unroll
                for (int i = 0; i < 5; ++i) m[i] = kRel<T> ? mp[i] + (xc[i] - xn[i]) : mp[i];   // from the next nominal on
#pragma unroll
                for (int i = 0; i < 15; ++i) P[i] = Pp[i];
            }
            if (!use_lin) sc = sn;
#pragma unroll
            for (int i = 0; i < 5; ++i) xc[i] = xn[i];
        }
        if (use_lin) {
            __syncwarp();   // every lane is done with the stage: refill it
            if (s + ST < steps) ws.issue(lin_warp<K>(p, s + ST, lane), st);
        }
    }
    if (use_lin) wpar = ws.parity;
    stores_before_bulk_reads();   // the RTS pass streams the filtered moments, after the grid barrier's block barrier
    return ok;
}

// The same over given arrays, with the log-likelihoods if they are wanted.
template <bool IP, typename T>
PES_DEV bool rerun_filter_arrays(const KParams<T>& p, int64_t a, int64_t e, int lane, int steps, const Gauss<T>& G, T* wstage,
                                 uint64_t* wbar, uint32_t& wpar)
{
    bool ok = true;
    LogLik<T> ll;   // of the measurements of trajectory llb in the chunk
    int llb = -1;
    SegCursor cur;
    if (a < e) cur.init(p.offsets, p.B, a);
    T m[5], P[15];
#pragma unroll
    for (int i = 0; i < 5; ++i) m[i] = G.m[i] + G.r[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) P[i] = G.P[i];
    FilterStream<T> ws;
    ws.init(wstage, wbar, wpar);
    if (!IP) ws.issue(array_warp<kFilterIn>(p, 0, lane), 0);
    if (!IP && steps > 1) ws.issue(array_warp<kFilterIn>(p, 1, lane), 1);
    int st = 0;
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
        const int64_t k = a + s;
        const int other = st == 0 ? 2 : st - 1;   // the stage of steps s - 1 and s + 2
        if (!IP) ws.wait(st, p.status);
        const bool head = k < e && (cur.forward(k), cur.is_head(k));
        T mp[5], Pp[15];
        if (k < e && !head) {
            Trans<T> tr;
            if (!IP && s > 0) array_trans(ws, other, tr);
            else load_array_trans<IP>(p, k, lane, tr);
            T FP[25];
            predict(tr, m, P, mp, FP, Pp);
        }
        if (!IP) __syncwarp();   // every lane is done with step s - 1
        if (!IP && s + 2 < steps) ws.issue(array_warp<kFilterIn>(p, s + 2, lane), other);
        if (k < e) {
            if (head) {
                load_prior(p, cur.b, m, P);
            } else {
                Obs<T> ob;
                if constexpr (IP) array_obs(ArrayState<T, kFilterIn>{p, k}, 0, ob);
                else array_obs(ws, st, ob);
                if (p.loglik) {
                    if (cur.b != llb) {
                        if (llb >= 0) atomicAdd(p.loglik + llb, ll.value());
                        ll = LogLik<T>();
                        llb = cur.b;
                    }
                    ok &= kf_update(ob, mp, Pp, m, P, &ll);
                } else {
                    ok &= kf_update(ob, mp, Pp, m, P);
                }
            }
            store_filtered(p, array_ix<IP>(p, k, s, lane), m, P);
        }
        st = st == 2 ? 0 : st + 1;
    }
    if (!IP) {
        __syncwarp();
        wpar = ws.parity;
    }
    if (llb >= 0) atomicAdd(p.loglik + llb, ll.value());
    return ok;
}

// The smoothing element of a lane's whole chunk [a, e), from the state at e to
// the state at a: Eq. 17 for the chunk as one transition. G is the predicted
// Gaussian at a, f the chunk's filtering element. Conditioned on the chunk's
// measurements, x_a - xr ~ N(d + D (eta - J d), D) with D = (P^{-1} + J)^{-1} and d
// the Gaussian's mean less xr, and x_e given x_a is (A, b, C). A trajectory that
// ends within the chunk cuts the element (E = 0); the state before a trajectory's
// first one ignores it.
template <typename T>
PES_DEV bool chunk_selem(const KParams<T>& p, int64_t a, int64_t e, const FElem<T>& f, const Gauss<T>& G,
                         SElem<T>& el)
{
    selem_identity(el);
    if (a >= e) return true;
    SegCursor cur;
    cur.init(p.offsets, p.B, a);
    if (cur.is_head(a)) {
        T z[15];
#pragma unroll
        for (int i = 0; i < 15; ++i) z[i] = T(0);
        selem_last(el, z, z);
        return true;
    }
    T D[15], dm[5], u[5], Du[5], md[5], ref[5];
    info_update_cov(G.P, f.J, D);
#pragma unroll
    for (int i = 0; i < 5; ++i) dm[i] = G.m[i] + (G.r[i] - f.xr[i]);
    sv(f.J, dm, u);
#pragma unroll
    for (int i = 0; i < 5; ++i) u[i] = f.eta[i] - u[i];
    sv(D, u, Du);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        dm[i] += Du[i];
        md[i] = kRel<T> ? dm[i] : G.m[i] + Du[i];   // from xr, or absolute
    }
    if (kRel<T>) {
        felem_ref(f, ref);
        selem_set_refs(el, ref, f.xr);
    }
    if (cur.next <= e) {
        selem_last(el, md, D);
        return true;
    }
    T mp[5], AD[25], Pp[15];
    mv(f.A, dm, mp);
#pragma unroll
    for (int i = 0; i < 5; ++i) mp[i] += f.b[i];
    m_s(f.A, D, AD);
    abt_sym_add(AD, f.A, f.C, Pp);
    return selem_from_prediction(md, D, AD, Pp, mp, el);
}

// The smoothing element of a state from stage i of the given arrays' stream (or from
// the arrays in place).
template <typename T, class S>
PES_DEV bool array_selem(const S& ws, int i, bool tail, SElem<T>& el)
{
    T m[5], P[15];
#pragma unroll
    for (int c = 0; c < 5; ++c) m[c] = ws.get(i, 45 + c);
#pragma unroll
    for (int c = 0; c < 15; ++c) P[c] = ws.get(i, 50 + c);
    if (tail) {
        selem_last(el, m, P);
        return true;
    }
    Trans<T> tr;
    array_trans(ws, i, tr);
    T mp[5], FP[25], Pp[15];
    predict(tr, m, P, mp, FP, Pp);
    return selem_from_prediction(m, P, FP, Pp, mp, el);
}

// IP: the elements themselves are kept for the RTS pass, [step][component][lane], each
// written and read by its own lane (50 scalars; forming one again costs more than
// they do where the arrays are read in place).
template <typename T, typename F>
PES_DEV void each_selem_scalar(const KParams<T>& p, int s, int lane, SElem<T>& el, F f)
{
    static_assert(LINS >= 50, "the scratch holds an element per state");
    T* q = p.lin + (size_t)s * 50 * p.NL + lane;
#pragma unroll
    for (int i = 0; i < 25; ++i) f(el.E[i], q[(size_t)i * p.NL]);
#pragma unroll
    for (int i = 0; i < 5; ++i) f(el.g[i], q[(size_t)(25 + i) * p.NL]);
#pragma unroll
    for (int i = 0; i < 15; ++i) f(el.L[i], q[(size_t)(30 + i) * p.NL]);
#pragma unroll
    for (int i = 0; i < 5; ++i) f(el.xr[i], q[(size_t)(45 + i) * p.NL]);
}

// Smoothing, level 1 in MODE_SMOOTH: fold the chunk's smoothing elements from
// the given filtered moments and transitions.
template <bool IP, typename T>
PES_DEV bool fold_smoother_arrays(const KParams<T>& p, int64_t a, int64_t e, int lane, int steps, SElem<T>& accS, T* wstage,
                                  uint64_t* wbar, uint32_t& wpar)
{
    bool ok = true;
    selem_identity(accS);
    SegCursor cur;
    if (a < e) cur.init(p.offsets, p.B, a);
    SmoothStream<T> ws;
    ws.init(wstage, wbar, wpar);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        if (!IP && i < steps) ws.issue(array_warp<kSmoothIn>(p, i, lane), i);
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
        if (!IP) ws.wait(s & 1, p.status);
        if (a + s < e) {
            cur.forward(a + s);
            SElem<T> el;
            if constexpr (IP) {
                ok &= array_selem(ArrayState<T, kSmoothIn>{p, a + s}, 0, cur.is_tail(a + s), el);
                each_selem_scalar(p, s, lane, el, [](T v, T& kept) { kept = v; });
            } else {
                ok &= array_selem(ws, s & 1, cur.is_tail(a + s), el);
            }
            combine_smoother(accS, el, accS);
        }
        if (IP) continue;
        __syncwarp();
        if (s + 2 < steps) ws.issue(array_warp<kSmoothIn>(p, s + 2, lane), s & 1);
    }
    if (!IP) wpar = ws.parity;
    return ok;
}

// Smoothing, level 5 in MODE_SMOOTH.
template <bool IP, typename T>
PES_DEV bool rts_arrays(const KParams<T>& p, int64_t a, int64_t e, int lane, int steps, const Gauss<T>& G, T* wstage,
                        uint64_t* wbar, uint32_t& wpar)
{
    bool ok = true;
    SegCursor cur;
    if (a < e) cur.init(p.offsets, p.B, e - 1);
    Gauss<T> s = G;
#pragma unroll
    for (int i = 0; i < 5; ++i) s.m[i] += G.r[i];
    SmoothStream<T> ws;
    ws.init(wstage, wbar, wpar);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        if (!IP && i < steps) ws.issue(array_warp<kSmoothIn>(p, steps - 1 - i, lane), i);
    int st = 0;
#pragma unroll 1
    for (int sidx = steps - 1; sidx >= 0; --sidx, st ^= 1) {
        const int64_t k = a + sidx;
        if (!IP) ws.wait(st, p.status);
        if (k < e) {
            cur.backward(k);
            const int64_t ix = array_ix<IP>(p, k, sidx, lane);
            SElem<T> el;
            if constexpr (IP) each_selem_scalar(p, sidx, lane, el, [](T& v, T kept) { v = kept; });
            else ok &= array_selem(ws, st, cur.is_tail(k), el);
            apply_smoother(el, s, s);
            bool finite = true;
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                finite = finite && isfinite(s.m[i]);
                p.x[i * p.cs + ix] = s.m[i];
            }
            if (!finite) atomicOr(p.status, ST_NONFINITE);
#pragma unroll
            for (int i = 0; i < 15; ++i) p.P[i * p.cs + ix] = s.P[i];
        }
        if (IP) continue;
        __syncwarp();
        if (sidx >= 2) ws.issue(array_warp<kSmoothIn>(p, sidx - 2, lane), st);
    }
    if (!IP) wpar = ws.parity;
    return ok;
}

// Smoothing, level 5: Rauch-Tung-Striebel re-run backwards from the Gaussian of
// the state after the chunk: x_k ~ E_k (x_{k+1} - xr_k) + g_k with covariance
// E P E^T + L (a last state has E = 0), each element built from the state's
// filtered moments and its outgoing transition. The filtered moments (and the
// stored linearisation, if any) arrive through a warp stream and the smoothed
// moments replace the nominal in place.
template <int K, typename T>
PES_DEV bool rts_chunk(const KParams<T>& p, int64_t a, int64_t e, int lane, int steps, const Gauss<T>& G, bool write_P,
                       bool want_norm, double* conv, int& nb, double& num, double& den, T* wstage, uint64_t* wbar,
                       uint32_t& wpar)
{
    constexpr int LIN = kLinOf<K>, FS = kFS<K>;
    bool ok = true;
    const bool any = a < e;
    SegCursor cur;
    if (any) cur.init(p.offsets, p.B, e - 1);
    Gauss<T> s = G;
    constexpr bool use_lin = kStoreLin<K>;
    constexpr int ST = kRtsStages<K>;
    WarpStream<T, HAND + (use_lin ? kLinTrans<K> : 0), ST> ws;
    const T* hand = p.hand + (size_t)(lane >> 5) * p.L * (HAND * 32);
    auto issue = [&](int sidx, int st) {
        if (use_lin) ws.issue2(hand + (size_t)sidx * (HAND * 32), HAND, lin_warp<K>(p, sidx, lane) + kLinTransAt<K> * 32,
                               kLinTrans<K>, st);
        else ws.issue(hand + (size_t)sidx * (HAND * 32), st);
    };
    ws.init(wstage, wbar, wpar);
#pragma unroll
    for (int i = 0; i < ST; ++i)
        if (i < steps) issue(steps - 1 - i, i);
    // the nominal a step ahead
    T xc[5], xn[5];   // nominals of states k, k-1
    if (any) {
        load_nominal(p, lane_ix(p, e - 1 - a, lane), xc);
#pragma unroll
        for (int c = 0; c < 5 && kRel<T>; ++c) s.m[c] += G.r[c] - xc[c];
    }
    int st = 0;
#pragma unroll 1
    for (int sidx = steps - 1; sidx >= 0; --sidx) {
        const int64_t k = a + sidx;
        ws.wait(st, p.status);
        if (k < e) {
            cur.backward(k);
            const int64_t ix = lane_ix(p, sidx, lane);
            if (k > a) load_nominal(p, ix - p.NL, xn);
            T m[5], P[15];
#pragma unroll
            for (int c = 0; c < 5; ++c) m[c] = ws.get(st, c);
#pragma unroll
            for (int c = 0; c < 15; ++c) P[c] = ws.get(st, 5 + c);
            if (cur.is_tail(k)) {
#pragma unroll
                for (int c = 0; c < 5; ++c) s.m[c] = m[c];
#pragma unroll
                for (int c = 0; c < 15; ++c) s.P[c] = P[c];
            } else {
                Trans<T> tr;
                if constexpr (use_lin) {
                    trans_from_stage<K>(p, ws, st, HAND - kLinTransAt<K>, xc, tr);
                } else {
                    StateIn<T, LIN> in;
                    Factor<T, LIN> fc;
#pragma unroll
                    for (int c = 0; c < 5; ++c) in.x[c] = xc[c];
                    form_trans<K>(p, in, fc, tr);
                }
                T mp[5], FP[25], Pp[15];
                predict<FS, kRel<T>>(tr, m, P, mp, FP, Pp);
                SElem<T> ec;
                ok &= selem_from_prediction(m, P, FP, Pp, mp, ec);
                apply_smoother(ec, s, s);
            }
            bool finite = true;
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                finite = finite && isfinite(s.m[i]);
                p.x[i * p.cs + ix] = kRel<T> ? xc[i] + s.m[i] : s.m[i];
            }
            if (!finite) atomicOr(p.status, ST_NONFINITE);
            if (write_P) {
#pragma unroll
                for (int i = 0; i < 15; ++i) p.P[i * p.cs + ix] = s.P[i];
            }
            if (want_norm) {
                if (cur.b != nb) {
                    if (nb >= 0) {
                        atomicAdd(conv + 2 * nb, num);
                        atomicAdd(conv + 2 * nb + 1, den);
                    }
                    nb = cur.b;
                    num = 0.0;
                    den = 0.0;
                }
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    const T x = kRel<T> ? xc[i] + s.m[i] : s.m[i];
                    const double dv = double(x) - double(xc[i]);
                    num += dv * dv;
                    den += double(x) * double(x);
                }
            }
#pragma unroll
            for (int c = 0; c < 5; ++c) {   // from the nominal of k - 1 on
                if (kRel<T>) s.m[c] += xc[c] - xn[c];
                xc[c] = xn[c];
            }
        }
        __syncwarp();   // every lane is done with the stage: refill it
        if (sidx >= ST) issue(sidx - ST, st);
        st = st + 1 == ST ? 0 : st + 1;
    }
    wpar = ws.parity;
    return ok;
}

// ---- block and grid levels -------------------------------------------------------------

// Lane t's element into the tree's leaves, and the tree's up-sweep; the block's
// element goes to slot `agg`.
template <typename T, int NT, class Ops, typename Elem>
PES_DEV void publish_block(const Elem& el, int nl, T* agg)
{
    constexpr int NC = Ops::NC;
    static_assert(sizeof(Elem) == NC * sizeof(T), "the element's scalars");
    const int t = threadIdx.x;
    T* s = smem_as<T>();
    if (t < nl) reinterpret_cast<Elem*>(s)[tree_place(t, nl)] = el;
    __syncthreads();
    const int root = tree_reduce<T, NT, Ops>(0, -1, nl);
    for (int c = t; c < NC; c += NT) agg[c] = s[root + c];
}

template <typename T, int K, int NT>
constexpr size_t smem_bytes_for()
{
    using M = TreeMem<T, NT>;
    static_assert(M::kEnd - FE * NT >= NT * 3 * kStateIn, "the sigma-point folds' prefetch fits beside the leaves");
    static_assert(!kArrays<K> || (M::kEnd - FE * NT >= NT * 2 * kFilterIn && M::kEnd >= NT * 3 * kFilterIn &&
                                     M::kEnd - SE * NT >= NT * 2 * kSmoothIn),
                  "the streams of the scans over given arrays fit");
    static_assert(M::kBlock - M::kAfterSmootherTree >= NT * kLinStages<K> * kLinScalars<K>, "the re-run's stages fit");
    static_assert(M::kEnd >= NT * kRtsStages<K> * (HAND + (kStoreLin<K> ? kLinTrans<K> : 0)), "the RTS stages fit");
    static_assert(M::kEnd >= 2 * NT * int(sizeof(double) / sizeof(T)), "the norm reduction fits");
    return sizeof(T) * M::kEnd;
}

template <typename T, int K, int NT>
__global__ void __launch_bounds__(NT, 1) pes_persistent_kernel(const KParams<T> p)
{
    using M = TreeMem<T, NT>;
    T* smem = smem_as<T>();
    __shared__ int s_flag;
    // per-warp stream stages reuse the tree memory during the sequential passes
    __shared__ __align__(8) uint64_t s_bar[kMaxStages * (NT / 32)];
    const int warp = threadIdx.x >> 5;
    uint64_t* wbar = s_bar + kMaxStages * warp;
    uint32_t wpar = 0;
    if ((threadIdx.x & 31) == 0)
        for (int i = 0; i < kMaxStages; ++i) mbar_init(wbar + i, 1);
    mbar_init_fence();
    __syncthreads();

    const int t = threadIdx.x;
    // the block's first lpb threads, whole warps, are lanes; the others help with
    // the trees only
    const int lane = blockIdx.x * p.lpb + t;
    const int steps = t < p.lpb ? p.L : 0;
    const int64_t a = steps ? min((int64_t)lane * p.L, p.N) : p.N;
    const int64_t e = min(a + (int64_t)p.L, p.N);
    // lanes of this block with a chunk (its first ones); one identity if none
    const int nl = (int)max((int64_t)1, min((int64_t)p.lpb, (p.N + p.L - 1) / p.L - (int64_t)blockIdx.x * p.lpb));
    unsigned gen = 0;
    bool ok = true;

    const bool do_filter = (p.mode != MODE_SMOOTH);
    const bool do_smooth = (p.mode != MODE_FILTER);
    const bool track = (p.mode == MODE_RUN) && (p.tol > 0.0);

    int it = 0;
    bool converged = false;
#pragma unroll 1
    for (it = 0; it < p.iters; ++it) {
        // another block may set the bit while this one reads it: one answer for all
        // its threads, which meet at barriers from here on
        if (__syncthreads_or(*(volatile int*)p.status & (ST_TIMEOUT | ST_BADARG))) break;
        const bool last = (it == p.iters - 1);
        T* aggF = p.aggF + (size_t)(it & 1) * p.agg_blocks * FE;
        T* aggS = p.aggS + (size_t)(it & 1) * p.agg_blocks * SE;
        PES_PHASE(p, it, 0);
        SElem<T> accS;
        Gauss<T> G;
        using Ops = std::conditional_t<kKeepRounding<K, T>, FilterOps1<T>, FilterOps<T>>;
        using SOps = std::conditional_t<kKeepRounding<K, T>, SmootherOps1<T>, SmootherOps<T>>;
        if (do_filter) {
            FElem<T> acc;
            // the fold's prefetch goes to memory beside the leaves
            if constexpr (kArrays<K>)
                ok &= fold_filter_arrays<K == KK_ARRAYS_IN_PLACE>(p, a, e, lane, steps, acc, smem + FE * NT + (size_t)warp * 2 * kFilterIn * 32, wbar, wpar);
            else
                ok &= fold_filter_chunk<K>(p, a, e, lane, acc, Prefetch<T, kStateIn>{smem + FE * NT + t, NT, p.x, p.cs});
            PES_PHASE(p, it, 1);
            publish_block<T, NT, Ops>(acc, nl, aggF + (size_t)blockIdx.x * FE);
            PES_PHASE(p, it, 2);
            grid_arrive(p, gen);
            grid_wait(p, gen);
            PES_PHASE(p, it, 3);
            tree_top<T, NT, Ops>(aggF, 0, blockIdx.x);
            PES_PHASE(p, it, 4);
            tree_down<T, NT, Ops>(nl);
            G = reinterpret_cast<const Gauss<T>*>(smem + M::kGauss)[min(t, nl - 1)];
            PES_PHASE(p, it, 5);
            if (do_smooth) ok &= chunk_selem(p, a, e, reinterpret_cast<const FElem<T>*>(smem)[tree_place(min(t, nl - 1), nl)], G, accS);
        } else {
            if constexpr (kArrays<K>)
                ok &= fold_smoother_arrays<K == KK_ARRAYS_IN_PLACE>(p, a, e, lane, steps, accS, smem + SE * NT + (size_t)warp * 2 * kSmoothIn * 32, wbar, wpar);
        }
        __syncthreads();   // the smoother's tree and the stream stages overlap the filter's
        if (do_smooth) {
            publish_block<T, NT, SOps>(accS, nl, aggS + (size_t)blockIdx.x * SE);
            grid_arrive(p, gen);
        }
        PES_PHASE(p, it, 6);
        if (do_filter) {
            if constexpr (kArrays<K>) {
                ok &= rerun_filter_arrays<K == KK_ARRAYS_IN_PLACE>(p, a, e, lane, steps, G, smem + (size_t)warp * 3 * kFilterIn * 32, wbar, wpar);
            } else {
                constexpr int kStage = kLinStages<K> * kLinScalars<K> * 32;
                ok &= rerun_filter_chunk<K>(p, a, e, lane, steps, G, smem + M::kAfterSmootherTree + (size_t)warp * kStage, wbar, wpar);
            }
            if (track && blockIdx.x == 0) {
                // the accumulators of the next iteration were last read before
                // this iteration's first barrier; clear them for reuse
                double* nxt = p.conv + (size_t)((it + 1) & 1) * 2 * p.B;
                for (int i = t; i < 2 * p.B; i += NT) nxt[i] = 0.0;
            }
        }
        PES_PHASE(p, it, 7);
        if (do_smooth) {
            grid_wait(p, gen);
            PES_PHASE(p, it, 8);
            tree_top<T, NT, SOps>(aggS, blockIdx.x + 1, gridDim.x);
            PES_PHASE(p, it, 9);
            tree_down<T, NT, SOps>(nl);
            const Gauss<T> Gs = reinterpret_cast<const Gauss<T>*>(smem + M::kGauss)[min(t, nl - 1)];
            __syncthreads();   // the stream stages overlap the tree
            PES_PHASE(p, it, 10);
            const bool write_P = kSigma<kLinOf<K>> || last || p.write_P_every_iter;
            int nb = -1;
            double num = 0.0, den = 0.0;
            double* conv = p.conv + (size_t)(it & 1) * 2 * p.B;
            if constexpr (kArrays<K>) {
                ok &= rts_arrays<K == KK_ARRAYS_IN_PLACE>(p, a, e, lane, steps, Gs, smem + (size_t)warp * 2 * kSmoothIn * 32, wbar, wpar);
            } else {
                constexpr int kStage = kRtsStages<K> * (HAND + (kStoreLin<K> ? kLinTrans<K> : 0)) * 32;
                ok &= rts_chunk<K>(p, a, e, lane, steps, Gs, write_P, track, conv, nb, num, den, smem + (size_t)warp * kStage, wbar, wpar);
            }
            __syncthreads();
            PES_PHASE(p, it, 11);
            if (track && nb >= 0) {
                atomicAdd(conv + 2 * nb, num);
                atomicAdd(conv + 2 * nb + 1, den);
            }
        }
        if (track) {
            grid_arrive(p, gen);
            grid_wait(p, gen);
            PES_PHASE(p, it, 12);
            {
                // worst relative update norm over trajectories, identical in every block
                const double* conv = p.conv + (size_t)(it & 1) * 2 * p.B;
                double worst = 0.0;
                for (int b = t; b < p.B; b += NT) {
                    const double num = __ldcg(conv + 2 * b), den = __ldcg(conv + 2 * b + 1);
                    const double r = den > 0.0 ? sqrt(num / den) : sqrt(num);
                    worst = fmax(worst, r);
                    if (p.traj_iters && blockIdx.x == 0 && r <= p.tol && p.traj_iters[b] == 0) p.traj_iters[b] = it + 1;
                }
                double* s_red = reinterpret_cast<double*>(smem);   // the sequential passes are over
                s_red[t] = worst;
                __syncthreads();
                for (int s = NT / 2; s > 0; s >>= 1) {
                    if (t < s) s_red[t] = fmax(s_red[t], s_red[t + s]);
                    __syncthreads();
                }
                if (t == 0) s_flag = (s_red[0] <= p.tol) ? 1 : 0;
                __syncthreads();
                const int done = s_flag;
                __syncthreads();
                if (done) {
                    converged = true;
                    ++it;
                    break;
                }
            }
        }
    }
    if (!ok) atomicOr(p.status, ST_NOT_PD);
    if (blockIdx.x == 0 && t == 0) {
        if (p.iters_done) *p.iters_done = it;
        if (track && !converged) atomicOr(p.status, ST_NOT_CONVERGED);
    }
}

}  // namespace pes
