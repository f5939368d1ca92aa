// The block and grid levels of the scans: trees of elements in shared memory
// whose operators are each evaluated by several threads.
//
// What bounds a tree level is the latency of one operator: Eq. 15 is about
// 2,000 instructions on one thread, 4,480 cycles in FP32 and 103,000 in FP64
// (one warp, operands in shared memory), and a level of a 256-lane tree has
// 128, 64, ... 1 of them. Written for the rows of its outputs, Eq. 15 falls
// into eleven tasks of one form that share the factorisation of C_i and J_j:
//   t = a_r                 (row r of A_j):       row r of A and of C
//   t = J_j z_c             (z_c column c of A_i): column c of J
//   t = eta_j - J_j (b_i - xr_j):                 eta and b
//   p = D t,  w = t - J_j p,  o1 = A_i^T w,  o2 = A_j p
// with D = (C_i^{-1} + J_j)^{-1}. So a level's operators are spread over all
// the block's threads: operator i of m on threads i, i + m', i + 2 m', ...
// (m' >= m a power of two), each taking every (NT / m')-th task. The
// factorisation (about 260 instructions) is repeated in each of them, a task is
// about 130. The other operators are split by rows in the same way. (61 FP32
// lanes: up-sweep 15.7 -> 8.4 us, down-sweep 6.8 -> 4.8; 125 FP64 lanes: 50 -> 26
// us per level of the up-sweep, rsqrt pivots included.)
//
// Elements are stored whole (76 and 60 scalars, padded), one after another: the
// operands arrive in 16-byte loads, and at these strides consecutive elements'
// 16-byte words fall in different banks. Within a level the even nodes (left
// children) come first, then the odd ones, so that the operands of consecutive
// operators are consecutive elements. Every level is kept: the down-sweep needs
// the left (smoothing: right) children of each, the lanes their own element.
#pragma once

#include "pes_ops.cuh"

namespace pes {

constexpr int FE = sizeof(FElem<double>) / sizeof(double);   // 76
constexpr int SE = sizeof(SElem<double>) / sizeof(double);   // 60
constexpr int GE = sizeof(Gauss<double>) / sizeof(double);   // 28
// offsets of an element's fields
constexpr int FA = 0, FB = 25, FC = 32, FJ = 48, FETA = 64, FXR = 69;
constexpr int EE = 0, EG = 25, EL = 32, EXR = 48, EGR = 53;
constexpr int GR = 20;
// where entry q of a filtering element's output reference is, and of a smoothing
// element's input reference
PES_DEV int f_ref(int q) { return q < 2 ? 30 + q : (q == 2 ? 47 : (q == 3 ? 63 : 74)); }
PES_DEV int s_ref(int q) { return q < 2 ? 30 + q : (q == 2 ? 47 : 55 + q); }

// dynamic shared memory of the calling kernel, as scalars
template <typename T>
PES_DEV T* smem_as()
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    return reinterpret_cast<T*>(smem_raw);
}

// place of a packed symmetric matrix's row r: entry (r, c), c >= r, is at
// si_row(r, c) = si_row(r, 0) + c
PES_DEV int si_row(int r, int c) { return r * 5 - (r * (r - 1)) / 2 + (c - r); }

// N scalars (a multiple of 16 bytes) by 16-byte loads
template <int N>
PES_DEV void ld_vec(const float* s, float* r)
{
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
        const float4 v = reinterpret_cast<const float4*>(s)[i];
        r[4 * i] = v.x;
        r[4 * i + 1] = v.y;
        r[4 * i + 2] = v.z;
        r[4 * i + 3] = v.w;
    }
}
template <int N>
PES_DEV void ld_vec(const double* s, double* r)
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const double2 v = reinterpret_cast<const double2*>(s)[i];
        r[2 * i] = v.x;
        r[2 * i + 1] = v.y;
    }
}

// and by 16-byte stores
template <int N>
PES_DEV void st_vec(float* s, const float* r)
{
#pragma unroll
    for (int i = 0; i < N / 4; ++i)
        reinterpret_cast<float4*>(s)[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
}
template <int N>
PES_DEV void st_vec(double* s, const double* r)
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i) reinterpret_cast<double2*>(s)[i] = make_double2(r[2 * i], r[2 * i + 1]);
}

// The operators work on elements at offsets (in scalars) of shared memory: a, b
// the operands, o the result (another element), for the calling thread's tasks
// part, part + parts, ...

// o = a (x) b, Eq. 15. The first task's operands are loaded before the
// factorisation, which hides them; tasks differ only in addresses and selects.
template <typename T>
PES_DEV void coop_combine_filter(int a, int b, int o, int part, int parts)
{
    if (part >= 11) return;
    T* s = smem_as<T>();
    const T* pa = s + a;
    const T* pb = s + b;
    T* po = s + o;
    T J[16], D[15], C[16], off[5], eta[5], z[5], add[5];
    ld_vec<16>(pb + FJ, J);
    ld_vec<16>(pa + FC, C);
    int r, base;        // the packed row (column) of C (J) that the task writes, and its place
    bool row, vec;
    auto load_task = [&](int task) {
        row = task < 5;
        vec = task == 10;
        r = row ? task : (vec ? 0 : task - 5);
        const T* src = row ? pb + FA + 5 * task : (vec ? pa + FB : pa + FA + r);
        const int step = (row || vec) ? 1 : 5;
#pragma unroll
        for (int i = 0; i < 5; ++i) z[i] = src[i * step];
        base = vec ? FETA : (row ? FC + si_row(r, 0) : FJ + r);
        const T* q = row ? pb : pa;
        // entries (r, c) of a packed row, c >= r, or (c, r) of a packed column, c <= r
#pragma unroll
        for (int c = 0; c < 5; ++c) add[c] = q[base + ((row || vec) ? c : si(c, c) - c)];
    };
    load_task(part);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        off[i] = pa[f_ref(i)] - pb[FXR + i];   // where a's output is measured from, to b's input
        eta[i] = pb[FETA + i];
    }
    info_update_cov(C, J, D);
    T Ai[28], Aj[32];   // Aj: A then b
    ld_vec<28>(pa + FA, Ai);
    ld_vec<32>(pb + FA, Aj);
#pragma unroll 1
    for (int task = part;;) {
        T t[5], p[5], w[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) z[i] = vec ? z[i] + off[i] : z[i];
        sv(J, z, t);
#pragma unroll
        for (int i = 0; i < 5; ++i) t[i] = row ? z[i] : (vec ? eta[i] - t[i] : t[i]);
        sv(D, t, p);
        sv(J, p, w);
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = t[i] - w[i];
        T o1[5], o2[5];
        if (row || vec) {
            // A_i^T w: row r of A, or eta; A_j p (+ C), or A_j (z + p) + b
            mtv(Ai, w, o1);
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                const T start = vec ? Aj[c * 5] * (z[0] + p[0]) : fma(p[0], Aj[c * 5], add[c]);
                T v = start;
#pragma unroll
                for (int l = 1; l < 5; ++l) v = fma(vec ? z[l] + p[l] : p[l], Aj[c * 5 + l], v);
                o2[c] = v;
            }
            T* const oa = po + (vec ? FETA : FA + 5 * task);
            T* const oc = po + (vec ? FB : base);
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                oa[c] = vec ? o1[c] + add[c] : o1[c];
                if (c >= r) oc[c] = vec ? o2[c] + Aj[FB + c] : o2[c];
            }
        } else {
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                T v = add[c];
#pragma unroll
                for (int l = 0; l < 5; ++l) v = fma(Ai[l * 5 + c], w[l], v);
                if (c <= r) po[base + si(c, c) - c] = v;
            }
            po[FXR + r] = pa[FXR + r];
            po[f_ref(r)] = pb[f_ref(r)];
        }
        task += parts;
        if (task >= 11) break;
        load_task(task);
    }
}

// (m, P) at g pushed through the element at e into the Gaussian at o.
template <typename T>
PES_DEV void coop_apply_filter(int g, int e, int o, int part, int parts)
{
    if (part >= 5) return;
    T* s = smem_as<T>();
    const T* pe = s + e;
    T* po = s + o;
    T G[28], J[16], D[15], w[5], xr[5], eta[5], row[5], add[5], br, ref;
    ld_vec<28>(s + g, G);
    ld_vec<16>(pe + FJ, J);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        xr[i] = pe[FXR + i];
        eta[i] = pe[FETA + i];
    }
    int base;
    auto load_row = [&](int r) {
        base = si_row(r, 0);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            row[i] = pe[FA + 5 * r + i];
            add[i] = pe[FC + base + i];
        }
        br = pe[FB + r];
        ref = pe[f_ref(r)];
    };
    load_row(part);
    T A[28];
    ld_vec<28>(pe + FA, A);
    info_update_cov(G + 5, J, D);
    {
        T dm[5], u[5], Du[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) dm[i] = G[i] + (G[GR + i] - xr[i]);
        sv(J, dm, u);
#pragma unroll
        for (int i = 0; i < 5; ++i) u[i] = eta[i] - u[i];
        sv(D, u, Du);
#pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = dm[i] + Du[i];
    }
#pragma unroll 1
    for (int r = part;;) {
        T p[5];
        sv(D, row, p);
        T m = row[0] * w[0];
#pragma unroll
        for (int i = 1; i < 5; ++i) m = fma(row[i], w[i], m);
        po[r] = m + br;
        po[GR + r] = ref;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            T v = add[c];
#pragma unroll
            for (int l = 0; l < 5; ++l) v = fma(p[l], A[c * 5 + l], v);
            if (c >= r) po[5 + base + c] = v;
        }
        r += parts;
        if (r >= 5) break;
        load_row(r);
    }
}

// o = a (x) b, Eq. 19 (a earlier in time).
template <typename T>
PES_DEV void coop_combine_smoother(int a, int b, int o, int part, int parts)
{
    if (part >= 5) return;
    T* s = smem_as<T>();
    const T* pa = s + a;
    const T* pb = s + b;
    T* po = s + o;
    T Ei[28], Ej[32], Lj[16], dg[5];   // Ej: E then g
    ld_vec<28>(pa + EE, Ei);
    ld_vec<32>(pb + EE, Ej);
    ld_vec<16>(pb + EL, Lj);
#pragma unroll
    for (int i = 0; i < 5; ++i) dg[i] = (Ej[EG + i] - pa[EXR + i]) + (pb[EGR + i] - pa[s_ref(i)]);
#pragma unroll 1
    for (int r = part; r < 5; r += parts) {
        T e[5], add[5], le[5], en[5];
        const int base = EL + si_row(r, 0);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            e[i] = pa[EE + 5 * r + i];
            add[i] = pa[base + i];
        }
        const T gr = pa[EG + r], xr = pb[EXR + r], gref = pa[EGR + r], sref = pb[s_ref(r)];
        sv(Lj, e, le);
        mtv(Ej, e, en);
        T g = e[0] * dg[0];
#pragma unroll
        for (int i = 1; i < 5; ++i) g = fma(e[i], dg[i], g);
        po[EG + r] = g + gr;
        po[EXR + r] = xr;
        po[EGR + r] = gref;
        po[s_ref(r)] = sref;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            T v = add[c];
#pragma unroll
            for (int l = 0; l < 5; ++l) v = fma(le[l], Ei[c * 5 + l], v);
            po[EE + 5 * r + c] = en[c];
            if (c >= r) po[base + c] = v;
        }
    }
}

// The smoothing Gaussian at g pushed back through the element at e into o.
template <typename T>
PES_DEV void coop_apply_smoother(int g, int e, int o, int part, int parts)
{
    if (part >= 5) return;
    T* s = smem_as<T>();
    const T* pe = s + e;
    T* po = s + o;
    T E[28], G[28], dm[5];
    ld_vec<28>(pe + EE, E);
    ld_vec<28>(s + g, G);
#pragma unroll
    for (int i = 0; i < 5; ++i) dm[i] = (G[i] - pe[EXR + i]) + (G[GR + i] - pe[s_ref(i)]);
#pragma unroll 1
    for (int r = part; r < 5; r += parts) {
        T row[5], add[5], p[5];
        const int base = si_row(r, 0);
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            row[i] = pe[EE + 5 * r + i];
            add[i] = pe[EL + base + i];
        }
        const T gr = pe[EG + r], gref = pe[EGR + r];
        sv(G + 5, row, p);
        T m = row[0] * dm[0];
#pragma unroll
        for (int i = 1; i < 5; ++i) m = fma(row[i], dm[i], m);
        po[r] = m + gr;
        po[GR + r] = gref;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            T v = add[c];
#pragma unroll
            for (int l = 0; l < 5; ++l) v = fma(p[l], E[c * 5 + l], v);
            if (c >= r) po[5 + base + c] = v;
        }
    }
}

// The smoothing operators by one thread each, for the lower levels.
template <typename T>
PES_DEV void combine_smoother1(int a, int b, int o)
{
    T* s = smem_as<T>();
    const T* pa = s + a;
    const T* pb = s + b;
    // E then g and two of the input's reference; L and one more; xr, gr and the last two
    T Ei[32], Ej[32], Li[16], Lj[16], xi[12], xj[12], dg[5], out[32], EL_[25];
    ld_vec<32>(pa + EE, Ei);
    ld_vec<32>(pb + EE, Ej);
    ld_vec<16>(pa + EL, Li);
    ld_vec<16>(pb + EL, Lj);
    ld_vec<12>(pa + EXR, xi);
    ld_vec<12>(pb + EXR, xj);
    const T ri[5] = {Ei[30], Ei[31], Li[15], xi[10], xi[11]};
#pragma unroll
    for (int i = 0; i < 5; ++i) dg[i] = (Ej[EG + i] - xi[i]) + (xj[5 + i] - ri[i]);
    mv(Ei, dg, out + EG);
#pragma unroll
    for (int i = 0; i < 5; ++i) out[EG + i] += Ei[EG + i];
    out[30] = Ej[30];
    out[31] = Ej[31];
    mm(Ei, Ej, out);
    st_vec<32>(s + o + EE, out);
    m_s(Ei, Lj, EL_);
    abt_sym_add(EL_, Ei, Li, out);
    out[15] = Lj[15];
    st_vec<16>(s + o + EL, out);
#pragma unroll
    for (int i = 0; i < 5; ++i) xj[5 + i] = xi[5 + i];
    st_vec<12>(s + o + EXR, xj);
}

template <typename T>
PES_DEV void apply_smoother1(int g, int e, int o)
{
    T* s = smem_as<T>();
    const T* pe = s + e;
    T E[32], G[28], L[16], x[12], dm[5], EP[25], out[28];
    ld_vec<32>(pe + EE, E);
    ld_vec<28>(s + g, G);
    ld_vec<12>(pe + EXR, x);
    ld_vec<16>(pe + EL, L);
    const T ri[5] = {E[30], E[31], L[15], x[10], x[11]};
#pragma unroll
    for (int i = 0; i < 5; ++i) dm[i] = (G[i] - x[i]) + (G[GR + i] - ri[i]);
    mv(E, dm, out);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        out[i] += E[EG + i];
        out[GR + i] = x[5 + i];
    }
    out[25] = out[26] = out[27] = T(0);
    m_s(E, G + 5, EP);
    abt_sym_add(EP, E, L, out + 5);
    st_vec<28>(s + o, out);
}

// The filtering operators by one thread each, for means that are absolute: all
// reference points are zero, and the results' stay so.
template <typename T>
PES_DEV void combine_filter1(int a, int b, int o)
{
    T* s = smem_as<T>();
    const FElem<T> ai = *reinterpret_cast<const FElem<T>*>(s + a), aj = *reinterpret_cast<const FElem<T>*>(s + b);
    FElem<T> out = aj;
    combine_filter(ai, aj, out);
    *reinterpret_cast<FElem<T>*>(s + o) = out;
}

template <typename T>
PES_DEV void apply_filter1(int g, int e, int o)
{
    T* s = smem_as<T>();
    const FElem<T> el = *reinterpret_cast<const FElem<T>*>(s + e);
    Gauss<T> out = *reinterpret_cast<const Gauss<T>*>(s + g);
    apply_filter(out, el, out);
    *reinterpret_cast<Gauss<T>*>(s + o) = out;
}

// The operators of the two scans, for the tree code below. `wide`: more than 32
// operators; all threads of a warp then have the same part. (A form of Eq. 15
// by two threads in registers was 20 % faster than its tasks at such levels in
// isolation, and slower in the kernel, where its code is fetched afresh in every
// iteration: up-sweep 19.7 against 15.8 us at 256 FP32 lanes.)
template <typename T>
struct FilterOps {
    static constexpr int NC = FE, kMean = FB, kCov = FC;
    PES_DEV static int ref(int q) { return f_ref(q); }
    static constexpr bool kSuffix = false;   // the Gaussian enters at the left
    PES_DEV static void combine(int a, int b, int o, int part, int parts, bool) { coop_combine_filter<T>(a, b, o, part, parts); }
    PES_DEV static void apply(int g, int e, int o, int part, int parts, bool) { coop_apply_filter<T>(g, e, o, part, parts); }
};

// Those of the FP32 scans over given arrays: combine_filter's rounding to the bit,
// which the FP64 log-likelihoods beside their results show. One thread per operator:
// the tasks above, with J through J_j - J_j D J_j as that function has it, were slower
// (251 lanes: up-sweep 16.2 us, here 12.6, down-sweep 9.0, here 6.1; 61 lanes the same,
// 8.5 and 4.6), and tasks for the upper levels with this for the lower ones slower
// still, as each launch fetches the code of both anew (256 lanes: up-sweep 17 to 23 us).
template <typename T>
struct FilterOps1 : FilterOps<T> {
    PES_DEV static void combine(int a, int b, int o, int part, int, bool)
    {
        if (part == 0) combine_filter1<T>(a, b, o);
    }
    PES_DEV static void apply(int g, int e, int o, int part, int, bool)
    {
        if (part == 0) apply_filter1<T>(g, e, o);
    }
};

template <typename T>
struct SmootherOps {
    static constexpr int NC = SE, kMean = EG, kCov = EL;
    PES_DEV static int ref(int q) { return EGR + q; }
    static constexpr bool kSuffix = true;    // the Gaussian enters at the right
    PES_DEV static void combine(int a, int b, int o, int part, int parts, bool wide)
    {
        if (!wide) coop_combine_smoother<T>(a, b, o, part, parts);
        else if (part == 0) combine_smoother1<T>(a, b, o);
    }
    PES_DEV static void apply(int g, int e, int o, int part, int parts, bool wide)
    {
        if (!wide) coop_apply_smoother<T>(g, e, o, part, parts);
        else if (part == 0) apply_smoother1<T>(g, e, o);
    }
};

// The same for the smoothing scan over given arrays (256 lanes: down-sweep 4.8 us with
// tasks for the upper levels, here 3.5).
template <typename T>
struct SmootherOps1 : SmootherOps<T> {
    PES_DEV static void combine(int a, int b, int o, int part, int, bool)
    {
        if (part == 0) combine_smoother1<T>(a, b, o);
    }
    PES_DEV static void apply(int g, int e, int o, int part, int, bool)
    {
        if (part == 0) apply_smoother1<T>(g, e, o);
    }
};

// Shared memory of a block's scans, in scalars: the tree of every level, and the
// grid level's aggregates (up to TOPN blocks at a time) with a second,
// half-size buffer that its levels alternate with. The leaves' Gaussians take
// the grid level's memory when that is done. 225 KB at 256 FP32 or 128 FP64
// threads, which run one block per SM; 114 KB at 128 FP32 threads, two blocks.
template <typename T, int NT>
struct TreeMem {
    static constexpr int TOPN = (sizeof(T) == 4 && NT == 256) ? 152 : (sizeof(T) == 4 ? 80 : 76);
    static constexpr int kTop = FE * 2 * NT;
    static constexpr int kTop2 = kTop + FE * TOPN;
    static constexpr int kGauss = kTop;
    static constexpr int kBlock = kTop2 + FE * (TOPN / 2);   // the Gaussian entering the block
    static constexpr int kEnd = kBlock + GE;
    static_assert(FE * (TOPN + TOPN / 2) >= GE * NT, "the leaves' Gaussians fit");
    // smoothing's tree is smaller; memory from here to kBlock is free between
    // its up-sweep and its grid level
    static constexpr int kAfterSmootherTree = SE * 2 * NT;
};

// A level of n nodes holds its (n + 1) / 2 even ones first, then the odd ones;
// the level above it, of (n + 1) / 2 nodes, follows.
PES_DEV int tree_place(int i, int n) { return (i >> 1) + (i & 1) * ((n + 1) >> 1); }

// The product of n >= 1 elements, stored as a level from `src` on (scalars), by
// a tree of all the block's threads. The levels follow one another, or
// alternate between src and `alt` (>= 0). Returns the product's offset. One
// copy of the operator's code serves the lane tree and the grid level, so it
// stays in the instruction cache.
template <typename T, int NT, class Ops>
__device__ __noinline__ int tree_reduce(int src, int alt, int n)
{
    constexpr int NC = Ops::NC;
    const int t = threadIdx.x;
#pragma unroll 1
    while (n > 1) {
        const int ops = n >> 1, out = (n + 1) >> 1;
        const int lg = 32 - __clz(out - 1);   // 2^lg >= out
        const int i = t & ((1 << lg) - 1), part = t >> lg, parts = NT >> lg;
        const int next = alt >= 0 ? alt : src + n * NC;
        const int left = src + i * NC, dst = next + tree_place(i, out) * NC;
        if (i < ops) {
            Ops::combine(left, left + out * NC, dst, part, parts, lg >= 6);
        } else if (i < out) {   // an odd last node moves up as it is
            T* s = smem_as<T>();
            for (int c = part; c < NC; c += parts) s[dst + c] = s[left + c];
        }
        if (alt >= 0) alt = src;
        src = next;
        n = out;
        __syncthreads();
    }
    return src;
}

// Level 4: the Gaussian entering the block (kBlock) pushed down the tree over
// its n leaves to every leaf: filtering, the Gaussian before the leaf's span,
// kept at the span's first leaf on the way; smoothing, the one after it, at
// its last leaf.
template <typename T, int NT, class Ops>
PES_DEV void tree_down(int n)
{
    using M = TreeMem<T, NT>;
    constexpr int NC = Ops::NC;
    const int t = threadIdx.x;
    if (t < GE) {
        T* s = smem_as<T>();
        s[M::kGauss + (Ops::kSuffix ? n - 1 : 0) * GE + t] = s[M::kBlock + t];
    }
    __syncthreads();
    int top = 0, base = 0;   // level under the root, its first node
    while ((1 << (top + 1)) < n) base += (n + (1 << top) - 1) >> top, ++top;
    if (n == 1) return;
#pragma unroll 1
    for (int l = top; l >= 0; --l) {
        const int nodes = (n + (1 << l) - 1) >> l;   // at level l
        const int ops = nodes >> 1;                  // parents with both children
        const int lg = 32 - __clz(ops - 1);
        const int i = t & ((1 << lg) - 1), part = t >> lg, parts = NT >> lg;
        if (i < ops) {
            const int left = (base + i) * NC, right = left + ((nodes + 1) >> 1) * NC;
            const int first = i << (l + 1), mid = first + (1 << l);
            if (Ops::kSuffix) {
                const int last = min(first + (2 << l), n) - 1;
                Ops::apply(M::kGauss + last * GE, right, M::kGauss + (mid - 1) * GE, part, parts, lg >= 6);
            } else {
                Ops::apply(M::kGauss + first * GE, left, M::kGauss + mid * GE, part, parts, lg >= 6);
            }
        }
        if (l > 0) base -= (n + (1 << (l - 1)) - 1) >> (l - 1);
        __syncthreads();
    }
}

// Elements [0, n) of global memory into a level of n + shift nodes from dst on,
// as its nodes shift .. shift + n - 1: all the copies in flight at once.
template <typename T, int NT, int NC>
PES_DEV void level_copy_in(T* dst, const T* src, int n, int shift, int nodes)
{
    constexpr int V = 16 / sizeof(T), Q = NC / V;
    for (int q = threadIdx.x; q < n * Q; q += NT) {
        const int i = q / Q, k = q - i * Q;
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + tree_place(i + shift, nodes) * NC + k * V);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src + (size_t)i * NC + k * V) : "memory");
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

// Level 3: the Gaussian entering the block into kBlock, from the aggregates of
// blocks [b0, b1): their product starts with a prior (ends with a last state),
// so it is a Gaussian whatever precedes it: A = 0 and (b, C), or E = 0 and (g,
// L), with the references. Zero if there are none.
template <typename T, int NT, class Ops>
PES_DEV void tree_top(const T* agg, int b0, int b1)
{
    using M = TreeMem<T, NT>;
    constexpr int NC = Ops::NC, at = Ops::kMean, at2 = Ops::kCov;
    const int t = threadIdx.x;
    T* s = smem_as<T>();
    int root = -1;
    while (b0 < b1) {
        // TOPN nodes at a time, filtering the earliest blocks first, smoothing
        // the latest; the product so far is the first (last) node
        const int had = root >= 0;
        const int n = min(M::TOPN - had, b1 - b0);
        const int c0 = Ops::kSuffix ? b1 - n : b0;
        if (Ops::kSuffix) b1 -= n;
        else b0 += n;
        if (had) {
            const T v = t < NC ? s[root + t] : T(0);
            __syncthreads();
            if (t < NC) s[M::kTop + tree_place(Ops::kSuffix ? n : 0, n + 1) * NC + t] = v;
        }
        level_copy_in<T, NT, NC>(s + M::kTop, agg + (size_t)c0 * NC, n, Ops::kSuffix ? 0 : had, n + had);
        __syncthreads();
        root = tree_reduce<T, NT, Ops>(M::kTop, M::kTop2, n + had);
    }
    if (t < GE)
        s[M::kBlock + t] = root < 0 || t >= 25 ? T(0) : s[root + (t < 5 ? at + t : (t < GR ? at2 + t - 5 : Ops::ref(t - GR)))];
    __syncthreads();
}

}  // namespace pes
