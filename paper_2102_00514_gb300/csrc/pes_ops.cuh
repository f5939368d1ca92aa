// Filtering and smoothing elements and their associative operators (Sec. 4).
//
// Filtering element (Eqs. 12-14): the conditional density
//   p(x_k | y, x_in) = N(A (x_in - xr) + b, C)
// and the likelihood of the data given the input state in information form,
//   p(y | x_in) ∝ exp(-1/2 d^T J d + eta^T d),  d = x_in - xr.
// The input is measured from a reference point xr (the nominal state the
// element starts from); with xr = 0 this is exactly the paper's (A, b, C, eta, J).
//
// Smoothing element (Eqs. 16-18): p(x_k | y_{1:k}, x_next) = N(E (x_next - xr) + g, L).
//
// Operators: Eq. 15 (filtering) and Eq. 19 (smoothing). Eq. 15 is evaluated
// through the symmetric matrix D = (I + C_i J_j)^{-1} C_i = (C_i^{-1} + J_j)^{-1}
// (see info_update_cov), using (I + C_i J_j)^{-1} = I - D J_j and
// (I + J_j C_i)^{-1} = I - J_j D.
#pragma once

#include "pes_model.cuh"

namespace pes {

// Padded so that the fields that are loaded together start on 16 bytes, and
// to sizes at which consecutive elements' 16-byte words fall in different
// shared-memory banks (76, 60 and 28 words). The padding holds reference points:
// means are kept as small deviations from them, so that combining elements does
// not round positions of tens to thousands of units over and over. The filtering
// element's output mean is br + b (and its input is measured from xr); the
// smoothing element maps x_next to E (x_next - (sr + xr)) + gr + g.
template <typename T>
struct alignas(16) FElem {
    T A[25];
    T b[5];
    T br0[2];
    T C[15];
    T br2;
    T J[15];
    T br3;
    T eta[5];
    T xr[5];
    T br4;
    T pad;
};

template <typename T>
PES_DEV void felem_set_ref(FElem<T>& f, const T* r)
{
    f.br0[0] = r[0];
    f.br0[1] = r[1];
    f.br2 = r[2];
    f.br3 = r[3];
    f.br4 = r[4];
    f.pad = T(0);
}
template <typename T>
PES_DEV void felem_ref(const FElem<T>& f, T* r)
{
    r[0] = f.br0[0];
    r[1] = f.br0[1];
    r[2] = f.br2;
    r[3] = f.br3;
    r[4] = f.br4;
}

template <typename T>
struct alignas(16) SElem {
    T E[25];
    T g[5];
    T sr0[2];
    T L[15];
    T sr2;
    T xr[5];
    T gr[5];
    T sr3[2];
};

// References of the input (sr) and of g (gr).
template <typename T>
PES_DEV void selem_set_refs(SElem<T>& e, const T* sr, const T* gr)
{
    e.sr0[0] = sr[0];
    e.sr0[1] = sr[1];
    e.sr2 = sr[2];
    e.sr3[0] = sr[3];
    e.sr3[1] = sr[4];
#pragma unroll
    for (int i = 0; i < 5; ++i) e.gr[i] = gr[i];
}

template <typename T>
struct alignas(16) Gauss {
    T m[5];   // mean less r
    T P[15];
    T r[5];
    T pad[3];
};

// ---- products with a structured slope ------------------------------------------
//
// The coordinated turn's slopes have entries that are 0 or 1 whatever the state
// (f adds its increments to the positions and keeps the turn rate; bearings see
// only the position). With the model known at compile time those terms are left
// out: about 170 instead of 350 multiply-adds for a folded prediction, 230
// instead of 305 for the update. In finite arithmetic the results are the same
// to the bit, as a term 0 x or 1 x adds no rounding.

// C = F B
template <int FS, typename T>
PES_DEV void f_mm(const T* F, const T* B, T* C)
{
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            T s = T(0);
            bool first = true;
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                const int k = f_entry<FS>(i, l);
                if (k == 0) continue;
                if (first) s = k == 1 ? B[l * 5 + j] : F[i * 5 + l] * B[l * 5 + j];
                else s = k == 1 ? s + B[l * 5 + j] : fma(F[i * 5 + l], B[l * 5 + j], s);
                first = false;
            }
            C[i * 5 + j] = s;
        }
}

// C = F S, S symmetric packed
template <int FS, typename T>
PES_DEV void f_ms(const T* F, const T* S, T* C)
{
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            T s = T(0);
            bool first = true;
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                const int k = f_entry<FS>(i, l);
                if (k == 0) continue;
                if (first) s = k == 1 ? S[si(l, j)] : F[i * 5 + l] * S[si(l, j)];
                else s = k == 1 ? s + S[si(l, j)] : fma(F[i * 5 + l], S[si(l, j)], s);
                first = false;
            }
            C[i * 5 + j] = s;
        }
}

// Out (sym) = A F^T + Add (sym), product known to be symmetric
template <int FS, typename T>
PES_DEV void f_abt_sym_add(const T* A, const T* F, const T* Add, T* Out)
{
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = i; j < 5; ++j) {
            T s = Add[si(i, j)];
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                const int k = f_entry<FS>(j, l);
                if (k == 0) continue;
                s = k == 1 ? s + A[i * 5 + l] : fma(A[i * 5 + l], F[j * 5 + l], s);
            }
            Out[si(i, j)] = s;
        }
}

// y = F x
template <int FS, typename T>
PES_DEV void f_mv(const T* F, const T* x, T* y)
{
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        T s = T(0);
        bool first = true;
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            const int k = f_entry<FS>(i, l);
            if (k == 0) continue;
            if (first) s = k == 1 ? x[l] : F[i * 5 + l] * x[l];
            else s = k == 1 ? s + x[l] : fma(F[i * 5 + l], x[l], s);
            first = false;
        }
        y[i] = s;
    }
}

// out (2x5) = H S, S symmetric packed, H zero from column HC on
template <int HC, typename T>
PES_DEV void h_ms(const T* H, const T* S, T* out)
{
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            T s = H[r * 5] * S[si(0, j)];
#pragma unroll
            for (int l = 1; l < HC; ++l) s = fma(H[r * 5 + l], S[si(l, j)], s);
            out[r * 5 + j] = s;
        }
}

// out (2x2 sym) = A H^T + Add
template <int HC, typename T>
PES_DEV void h_abt_sym_add(const T* A, const T* H, const T* Add, T* out)
{
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int q = r; q < 2; ++q) {
            T s = Add[si2(r, q)];
#pragma unroll
            for (int l = 0; l < HC; ++l) s = fma(A[r * 5 + l], H[q * 5 + l], s);
            out[si2(r, q)] = s;
        }
}

// Identity of Eq. 15 with input reference xr: (A = I, b = xr, C = 0, eta = 0, J = 0).
template <typename T>
PES_DEV void felem_identity(FElem<T>& a, const T* xr)
{
    set_identity(a.A);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        a.b[i] = xr[i];
        a.eta[i] = T(0);
        a.xr[i] = xr[i];
    }
#pragma unroll
    for (int i = 0; i < 15; ++i) {
        a.C[i] = T(0);
        a.J[i] = T(0);
    }
    const T zero[5] = {T(0), T(0), T(0), T(0), T(0)};
    felem_set_ref(a, zero);
}

// The Levenberg-Marquardt damping of state k as a filtering element: the
// pseudo-measurement xbar = x_k + e, e ~ N(0, I / lambda), through an identity
// transition, about the reference xr = xbar: A = I, b = xbar, C = 0, eta = 0,
// J = lambda I. acc (x) damping adds the damping to the state acc ends at.
template <typename T>
PES_DEV void felem_damping(FElem<T>& a, const T* xbar, T lambda)
{
    set_identity(a.A);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        a.b[i] = xbar[i];
        a.eta[i] = T(0);
        a.xr[i] = xbar[i];
    }
#pragma unroll
    for (int i = 0; i < 15; ++i) {
        a.C[i] = T(0);
        a.J[i] = T(0);
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) a.J[si(i, i)] = lambda;
}

// a (x) a_0 where a_0 is the prior element (A = 0, b = m0, C = P0, eta = J = 0):
// the conditional density forgets its input; the likelihood stays.
template <typename T>
PES_DEV void felem_apply_prior(FElem<T>& a, const T* m0, const T* P0)
{
#pragma unroll
    for (int i = 0; i < 25; ++i) a.A[i] = T(0);
#pragma unroll
    for (int i = 0; i < 5; ++i) a.b[i] = m0[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) a.C[i] = P0[i];
}

// acc <- acc (x) a_k for the single-step element a_k of Eqs. 13-14 built from
// the transition (k-1 -> k) and the observation at k.
//
// a_k's J_k = G^T S^{-1} G has rank n_y, so the Woodbury identity turns the
// 5x5 inverse (I + C J_k)^{-1} of Eq. 15 into the 2x2 S^{-1}: the product is a
// Kalman predict + update of the affine conditional acc. Predict
//   A- = F A,  b- = fx + F (b - xn),  C- = F C F^T + Q',
// update with S = H C- H^T + R', K = C- H^T S^{-1}, G = H A-, v = r - H (b- - xn_k):
//   A = A- - K G,  b = b- + K v,  C = C- - K H C-,
// and the likelihood of y_k given the input accumulates
//   J += G^T S^{-1} G,  eta += G^T S^{-1} v.
// REL: means are measured from the nominal of the state that the linearisation
// is about, and tr.fx is f(xn) - xn (the smoother kernel; the caller re-references
// them from state to state). Otherwise means and tr.fx are absolute.
//
// The two halves are folded separately, which keeps the transition and the
// observation from being live together: the prediction through the transition,
// after which a describes x_k given the input, and the update with the
// observation at k.
template <int FS = FS_DENSE, bool REL = false, typename T>
PES_DEV void fold_predict(FElem<T>& a, const Trans<T>& tr)
{
    T Am[25];
    f_mm<FS>(tr.F, a.A, Am);
    T dv[5], bm[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) dv[i] = REL ? a.b[i] : a.b[i] - tr.xn[i];
    f_mv<FS>(tr.F, dv, bm);
#pragma unroll
    for (int i = 0; i < 5; ++i) bm[i] += tr.fx[i];
    T FC[25], Cm[15];
    f_ms<FS>(tr.F, a.C, FC);
    f_abt_sym_add<FS>(FC, tr.F, tr.Q, Cm);
#pragma unroll
    for (int i = 0; i < 25; ++i) a.A[i] = Am[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) a.b[i] = bm[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) a.C[i] = Cm[i];
}

template <int FS = FS_DENSE, bool REL = false, typename T>
PES_DEV bool fold_update(FElem<T>& a, const Obs<T>& ob)
{
    constexpr int HC = kHCols<FS>;
    const T* Am = a.A;
    const T* bm = a.b;
    const T* Cm = a.C;
    // H C-
    T HCm[10];
    h_ms<HC>(ob.H, Cm, HCm);
    T S[3];
    h_abt_sym_add<HC>(HCm, ob.H, ob.R, S);
    T Si[3];
    const bool ok = inv2_spd(S, Si);
    // K^T = S^{-1} H C-,  G = H A-,  v
    T KT[10], G[10], v[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            KT[r * 5 + j] = Si[si2(r, 0)] * HCm[j] + Si[si2(r, 1)] * HCm[5 + j];
            T s = ob.H[r * 5] * Am[j];
#pragma unroll
            for (int l = 1; l < HC; ++l) s = fma(ob.H[r * 5 + l], Am[l * 5 + j], s);
            G[r * 5 + j] = s;
        }
        T hv = ob.r[r];
#pragma unroll
        for (int l = 0; l < HC; ++l) hv = fma(-ob.H[r * 5 + l], REL ? bm[l] : bm[l] - ob.xn[l], hv);
        v[r] = hv;
    }
    T Anew[25], bnew[5], Cnew[15];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
#pragma unroll
        for (int j = 0; j < 5; ++j)
            Anew[i * 5 + j] = fma(-KT[5 + i], G[5 + j], fma(-KT[i], G[j], Am[i * 5 + j]));
        bnew[i] = fma(KT[5 + i], v[1], fma(KT[i], v[0], bm[i]));
    }
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = i; j < 5; ++j)
            Cnew[si(i, j)] = fma(-KT[5 + i], HCm[5 + j], fma(-KT[i], HCm[j], Cm[si(i, j)]));
#pragma unroll
    for (int i = 0; i < 25; ++i) a.A[i] = Anew[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) a.b[i] = bnew[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) a.C[i] = Cnew[i];
    // likelihood of y_k given the input
    T SiG[10], Siv[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int j = 0; j < 5; ++j) SiG[r * 5 + j] = Si[si2(r, 0)] * G[j] + Si[si2(r, 1)] * G[5 + j];
        Siv[r] = Si[si2(r, 0)] * v[0] + Si[si2(r, 1)] * v[1];
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) {
#pragma unroll
        for (int j = i; j < 5; ++j)
            a.J[si(i, j)] = fma(G[5 + i], SiG[5 + j], fma(G[i], SiG[j], a.J[si(i, j)]));
        a.eta[i] = fma(G[5 + i], Siv[1], fma(G[i], Siv[0], a.eta[i]));
    }
    return ok;
}

// out = ai (x) aj, Eq. 15 (ai earlier in time). aj's input reference is the
// point where ai's output is measured from. The elements' reference points are
// not looked at: b and xr count as they are (so do g and xr below).
template <typename T>
PES_DEV void combine_filter(const FElem<T>& ai, const FElem<T>& aj, FElem<T>& out)
{
    T bt[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) bt[i] = ai.b[i] - aj.xr[i];
    T D[15];
    info_update_cov(ai.C, aj.J, D);
    T AD[25];
    m_s(aj.A, D, AD);
    // W = A_j (I + C_i J_j)^{-1} = A_j - (A_j D) J_j
    T W[25];
    m_s(AD, aj.J, W);
#pragma unroll
    for (int i = 0; i < 25; ++i) W[i] = aj.A[i] - W[i];
    // mean: A_j (I + C_i J_j)^{-1} (bt + C_i eta_j) + b_j = A_j (bt + D u) + b_j, u = eta_j - J_j bt
    T u[5], Du[5], w[5], Aw[5];
    sv(aj.J, bt, u);
#pragma unroll
    for (int i = 0; i < 5; ++i) u[i] = aj.eta[i] - u[i];
    sv(D, u, Du);
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = bt[i] + Du[i];
    mv(aj.A, w, Aw);
    // likelihood: A_i^T (I - J_j D) u + eta_i
    T JDu[5], z[5], Az[5];
    sv(aj.J, Du, JDu);
#pragma unroll
    for (int i = 0; i < 5; ++i) z[i] = u[i] - JDu[i];
    mtv(ai.A, z, Az);
    // K2 = J_j - J_j D J_j
    T JD[25], K2[15];
    {
        T Df[25];
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int j = 0; j < 5; ++j) Df[i * 5 + j] = D[si(i, j)];
        s_m(aj.J, Df, JD);
    }
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = i; j < 5; ++j) {
            T s = aj.J[si(i, j)];
#pragma unroll
            for (int l = 0; l < 5; ++l) s = fma(-JD[i * 5 + l], aj.J[si(l, j)], s);
            K2[si(i, j)] = s;
        }
    T K2A[25];
    {
        T K2f[25];
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int j = 0; j < 5; ++j) K2f[i * 5 + j] = K2[si(i, j)];
        mm(K2f, ai.A, K2A);
    }
    // outputs are written last, so out may alias either input
    T Anew[25];
    mm(W, ai.A, Anew);
    T Cnew[15];
    abt_sym_add(AD, aj.A, aj.C, Cnew);
    T Jnew[15];
    atb_sym_add(ai.A, K2A, ai.J, Jnew);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        out.b[i] = Aw[i] + aj.b[i];
        out.eta[i] = Az[i] + ai.eta[i];
        out.xr[i] = ai.xr[i];
    }
#pragma unroll
    for (int i = 0; i < 25; ++i) out.A[i] = Anew[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) {
        out.C[i] = Cnew[i];
        out.J[i] = Jnew[i];
    }
}

// (m, P) (x) a: a Gaussian state before a's span, pushed through a. This is
// Eq. 15 with a left operand whose A, eta, J vanish (a filtering prefix that
// starts at a prior element): the Gaussian is conditioned on a's likelihood,
// D = (P^{-1} + J)^{-1}, mean m + D (eta - J m), then mapped by (A, b, C).
template <typename T>
PES_DEV void apply_filter(const Gauss<T>& g, const FElem<T>& a, Gauss<T>& out)
{
    T dm[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) dm[i] = g.m[i] - a.xr[i];
    T D[15];
    info_update_cov(g.P, a.J, D);
    T u[5], Du[5], w[5], Aw[5];
    sv(a.J, dm, u);
#pragma unroll
    for (int i = 0; i < 5; ++i) u[i] = a.eta[i] - u[i];
    sv(D, u, Du);
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = dm[i] + Du[i];
    mv(a.A, w, Aw);
    T AD[25];
    m_s(a.A, D, AD);
    T Pn[15];
    abt_sym_add(AD, a.A, a.C, Pn);
#pragma unroll
    for (int i = 0; i < 5; ++i) out.m[i] = Aw[i] + a.b[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) out.P[i] = Pn[i];
}

// ---- smoothing --------------------------------------------------------------------

template <typename T>
PES_DEV void selem_identity(SElem<T>& a)
{
    set_identity(a.E);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        a.g[i] = T(0);
        a.xr[i] = T(0);
    }
#pragma unroll
    for (int i = 0; i < 15; ++i) a.L[i] = T(0);
    const T zero[5] = {T(0), T(0), T(0), T(0), T(0)};
    selem_set_refs(a, zero, zero);
}

// Eq. 18: the last state of a trajectory, E = 0, g = x*, L = P*.
template <typename T>
PES_DEV void selem_last(SElem<T>& a, const T* xf, const T* Pf)
{
#pragma unroll
    for (int i = 0; i < 25; ++i) a.E[i] = T(0);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        a.g[i] = xf[i];
        a.xr[i] = T(0);
    }
#pragma unroll
    for (int i = 0; i < 15; ++i) a.L[i] = Pf[i];
}

// Eq. 17 from the predicted moments of x_{k+1}: FP = F_k P*_k, Pp = FP F^T + Q'_k,
// mp = F-prediction of x*_k:
//   E = P* F^T Pp^{-1},  L = P* - E F P*,
// and g = x*_k - E mp is kept as (g = x*_k, xr = mp), i.e. the element maps
// x_{k+1} to E (x_{k+1} - mp) + x*_k.
template <typename T>
PES_DEV bool selem_from_prediction(const T* xf, const T* Pf, const T* FP, const T* Pp, const T* mp, SElem<T>& a)
{
    T Lc[25], rd[5];
    const bool ok = chol_pd(Pp, Lc, rd);
    T Et[25];
#pragma unroll
    for (int i = 0; i < 25; ++i) Et[i] = FP[i];
    chol_solve_cols(Lc, rd, Et);   // Et = Pp^{-1} F P* = E^T
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = 0; j < 5; ++j) a.E[i * 5 + j] = Et[j * 5 + i];
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = i; j < 5; ++j) {
            T s = Pf[si(i, j)];
#pragma unroll
            for (int l = 0; l < 5; ++l) s = fma(-Et[l * 5 + i], FP[l * 5 + j], s);
            a.L[si(i, j)] = s;
        }
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        a.g[i] = xf[i];
        a.xr[i] = mp[i];
    }
    return ok;
}

// Predicted moments of the transition tr applied to (m, P): mp, FP = F P, Pp.
template <int FS = FS_DENSE, bool REL = false, typename T>
PES_DEV void predict(const Trans<T>& tr, const T* m, const T* P, T* mp, T* FP, T* Pp)
{
    T dx[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) dx[i] = REL ? m[i] : m[i] - tr.xn[i];
    f_mv<FS>(tr.F, dx, mp);
#pragma unroll
    for (int i = 0; i < 5; ++i) mp[i] += tr.fx[i];
    f_ms<FS>(tr.F, P, FP);
    f_abt_sym_add<FS>(FP, tr.F, tr.Q, Pp);
}

// Running log-likelihood of a trajectory's measurements: the sum over steps of
// log N(v; 0, S) = -1/2 (v^T S^{-1} v + log det S) - log 2 pi, every term in FP64.
// Bound by the FP64 pipe, which issues one instruction per warp every 64 cycles: a
// step takes about 18, of them 9 of the quotient. The determinants are multiplied
// up, their binary exponents kept apart by integer instructions, and one logarithm
// is taken at the end (a product is half an ulp of 1 off in a step, a logarithm per
// step was up to an ulp of its value, and made the filter scan's re-run 41 us at N =
// 128,128, FP32). A determinant that is negative or NaN makes the result NaN, as
// its own logarithm would.
template <typename T>
struct LogLik {
    double q = 0.0, det = 1.0;   // det in [1, 2), or 0, infinite or NaN
    int exponent = 0, steps = 0;
    // the exponent of a normal x out of it
    PES_DEV void split(double& x)
    {
        const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
        if (e > 0 && e < 0x7ff) {
            exponent += e - 1023;
            x = __hiloint2double((hi & 0x800fffff) | 0x3ff00000, __double2loint(x));
        }
    }
    PES_DEV void add(T s00, T s01, T s11, T v0, T v1)
    {
        ++steps;
        const double c00 = s00, c01 = s01, c11 = s11, c2 = T(-2) * s01, w0 = v0, w1 = v1;
        double d = fma(-c01, c01, c00 * c11);
        // v^T adj(S) v
        q += fma(w0, fma(c2, w1, c11 * w0), w1 * (c00 * w1)) / d;
        const int hi = __double2hiint(d);
        if (hi < 0 && d != 0.0) {   // not positive definite
            d = __longlong_as_double(0x7ff8000000000000LL);
        } else if ((hi & 0x7ff00000) == 0) {   // subnormal or zero
            d *= 18014398509481984.0;          // 2^54
            exponent -= 54;
        }
        split(d);
        det *= d;
        split(det);
    }
    PES_DEV double value() const
    {
        const double ln2 = 0.69314718055994530942, log_2pi = 1.8378770664093454836;
        return -0.5 * (q + (log(det) + exponent * ln2)) - steps * log_2pi;
    }
};

// Kalman update of (mp, Pp) with the observation ob: (m, P).
template <int FS = FS_DENSE, bool REL = false, typename T>
PES_DEV bool kf_update(const Obs<T>& ob, const T* mp, const T* Pp, T* m, T* P, LogLik<T>* loglik = nullptr)
{
    constexpr int HC = kHCols<FS>;
    T HP[10];
    h_ms<HC>(ob.H, Pp, HP);
    T S[3];
    h_abt_sym_add<HC>(HP, ob.H, ob.R, S);
    T Si[3];
    const bool ok = inv2_spd(S, Si);
    T KT[10], v[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int j = 0; j < 5; ++j) KT[r * 5 + j] = Si[si2(r, 0)] * HP[j] + Si[si2(r, 1)] * HP[5 + j];
        T hv = ob.r[r];
#pragma unroll
        for (int l = 0; l < HC; ++l) hv = fma(-ob.H[r * 5 + l], REL ? mp[l] : mp[l] - ob.xn[l], hv);
        v[r] = hv;
    }
    if (loglik) loglik->add(S[si2(0, 0)], S[si2(0, 1)], S[si2(1, 1)], v[0], v[1]);
#pragma unroll
    for (int i = 0; i < 5; ++i) m[i] = fma(KT[5 + i], v[1], fma(KT[i], v[0], mp[i]));
#pragma unroll
    for (int i = 0; i < 5; ++i)
#pragma unroll
        for (int j = i; j < 5; ++j)
            P[si(i, j)] = fma(-KT[5 + i], HP[5 + j], fma(-KT[i], HP[j], Pp[si(i, j)]));
    return ok;
}

// out = ai (x) aj, Eq. 19 (ai earlier in time):
// E = E_i E_j, g = E_i (g_j - xr_i) + g_i, L = E_i L_j E_i^T + L_i, xr = xr_j.
template <typename T>
PES_DEV void combine_smoother(const SElem<T>& ai, const SElem<T>& aj, SElem<T>& out)
{
    T dg[5], Eg[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) dg[i] = aj.g[i] - ai.xr[i];
    mv(ai.E, dg, Eg);
    T EL[25];
    m_s(ai.E, aj.L, EL);
    T Ln[15];
    abt_sym_add(EL, ai.E, ai.L, Ln);
    T En[25];
    mm(ai.E, aj.E, En);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        out.g[i] = Eg[i] + ai.g[i];
        out.xr[i] = aj.xr[i];
    }
#pragma unroll
    for (int i = 0; i < 25; ++i) out.E[i] = En[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) out.L[i] = Ln[i];
}

// a (x) (m, P): the smoothing distribution of the state after a's span pushed
// back through a: m' = E (m - xr) + g, P' = E P E^T + L.
template <typename T>
PES_DEV void apply_smoother(const SElem<T>& a, const Gauss<T>& g, Gauss<T>& out)
{
    T dm[5], Em[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) dm[i] = g.m[i] - a.xr[i];
    mv(a.E, dm, Em);
    T EP[25];
    m_s(a.E, g.P, EP);
    T Pn[15];
    abt_sym_add(EP, a.E, a.L, Pn);
#pragma unroll
    for (int i = 0; i < 5; ++i) out.m[i] = Em[i] + a.g[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) out.P[i] = Pn[i];
}

}  // namespace pes
