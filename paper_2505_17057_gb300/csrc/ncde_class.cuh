// ncde_class.cuh -- the NCDE node update in class form on node pairs (NcdeClass in mmfd_internal.h; the
// class sums and the pair arithmetic as in nse_class.cuh).
//
// A node sends a+ E_p +- a- O_p along each direction.  With alike axes every axis pair shares one even
// part and every diagonal pair another, and the odd parts are multiples of e_p . B(phi); both time
// levels' parts are added before the directions are formed, so that a direction costs one addition
// however many levels there are.  Where the axes also share the flux polynomial (SHARED), B is
// evaluated once, all axis pairs have the same odd part, and those of the diagonal pairs with
// components of unlike sign vanish.
#pragma once

#include "nse_class.cuh"

namespace mmfd {
inline namespace MMFD_PK_NS {

// The coefficients of one kernel as pairs.
template <typename T, int DIM, int NL, bool SHARED>
struct NcdePk {
    Pk<T> m2[5], fx[SHARED ? 1 : DIM][4];
    Pk<T> eP[NL][2], eM[NL][2], cP[NL], cM[NL];
    Pk<T> oA[NL], oD[NL];   // axis pairs: oB; diagonal pairs: oB (SHARED: twice that, the factor of B for like signs)
};

template <typename T, int DIM, int NL, bool SHARED>
NcdePk<T, DIM, NL, SHARED> ncde_pk(const NcdeClass<T>& c) {
    using P = Pk<T>;
    NcdePk<T, DIM, NL, SHARED> o;
    for (int k = 0; k < 5; ++k) o.m2[k] = P::fill(c.m2[k]);
    for (int a = 0; a < (SHARED ? 1 : DIM); ++a)
        for (int k = 0; k < 4; ++k) o.fx[a][k] = P::fill(c.flux[a][k]);
    for (int l = 0; l < NL; ++l) {
        for (int k = 0; k < 2; ++k) {
            o.eP[l][k] = P::fill(c.eP[l][k]);
            o.eM[l][k] = P::fill(c.eM[l][k]);
        }
        o.cP[l] = P::fill(c.cP[l]);
        o.cM[l] = P::fill(c.cM[l]);
        o.oA[l] = P::fill(c.oB[l][0]);
        o.oD[l] = P::fill(SHARED ? T(2) * c.oB[l][1] : c.oB[l][1]);
    }
    return o;
}

// A pair of nodes, or one node, evaluated: parts summed over the levels.
template <typename V, int DIM>
struct NcdeParts {
    V E0, E1, ctr;
    V A[DIM];        // axis odd parts a- O_a
    V D[DIM];        // general flux: the diagonal odd parts' components (D_a +- D_b); SHARED: D[0] the like-sign one
};

// One operand kind for pairs and single nodes (the halo columns).
template <typename T>
struct One {
    T v;
};
template <typename T> __device__ __forceinline__ One<T> pfma(One<T> a, One<T> b, One<T> c) { return {rfma(a.v, b.v, c.v)}; }
template <typename T> __device__ __forceinline__ One<T> pmul(One<T> a, One<T> b) { return {rmul(a.v, b.v)}; }
template <typename T> __device__ __forceinline__ One<T> padd(One<T> a, One<T> b) { return {radd(a.v, b.v)}; }
template <typename T> __device__ __forceinline__ One<T> psub(One<T> a, One<T> b) { return {rsub(a.v, b.v)}; }
template <typename V, typename T>
__device__ __forceinline__ V as(const Pk<T>& c) {
    if constexpr (std::is_same<V, Pk<T>>::value) return c;
    else return V{c.lo()};
}

// phi[l]: the stored values at the levels.
template <bool SHARED, int DIM, int NL, typename V, typename T>
__device__ __forceinline__ void ncde_eval(const NcdePk<T, DIM, NL, SHARED>& c, const V (&phi)[NL], NcdeParts<V, DIM>& o) {
#pragma unroll
    for (int l = 0; l < NL; ++l) {
        const V p = phi[l];
        V m2 = as<V, T>(c.m2[4]);
#pragma unroll
        for (int k = 3; k >= 0; --k) m2 = pfma(m2, p, as<V, T>(c.m2[k]));
        V B[SHARED ? 1 : DIM];
#pragma unroll
        for (int a = 0; a < (SHARED ? 1 : DIM); ++a) {
            B[a] = as<V, T>(c.fx[a][3]);
#pragma unroll
            for (int k = 2; k >= 0; --k) B[a] = pfma(B[a], p, as<V, T>(c.fx[a][k]));
        }
        auto acc = [&](V& s, const Pk<T>& w, V x) { s = l == 0 ? pmul(as<V, T>(w), x) : pfma(as<V, T>(w), x, s); };
        auto acc2 = [&](V& s, const Pk<T>& w, V x) { s = pfma(as<V, T>(w), x, s); };
        acc(o.E0, c.eP[l][0], p);
        acc2(o.E0, c.eM[l][0], m2);
        acc(o.E1, c.eP[l][1], p);
        acc2(o.E1, c.eM[l][1], m2);
        acc(o.ctr, c.cP[l], p);
        acc2(o.ctr, c.cM[l], m2);
        if constexpr (SHARED) {
            acc(o.A[0], c.oA[l], B[0]);
            acc(o.D[0], c.oD[l], B[0]);
        } else {
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                acc(o.A[a], c.oA[l], B[a]);
                acc(o.D[a], c.oD[l], B[a]);
            }
        }
    }
}

// a- O of the axis pair a, and E +- O of the diagonal pair of axes (a, b) with like (LIKE: e_a = e_b = 1)
// or unlike (e_a = -1, e_b = 1) signs, SIGN its direction.
template <bool SHARED, int A, int SIGN, typename V, int DIM>
__device__ __forceinline__ V ncde_axis(const NcdeParts<V, DIM>& o) {
    return SIGN > 0 ? padd(o.E0, o.A[SHARED ? 0 : A]) : psub(o.E0, o.A[SHARED ? 0 : A]);
}
template <bool SHARED, int A, int B, bool LIKE, int SIGN, typename V, int DIM>
__device__ __forceinline__ V ncde_diag(const NcdeParts<V, DIM>& o) {
    if constexpr (SHARED) {
        if constexpr (!LIKE) return o.E1;
        else return SIGN > 0 ? padd(o.E1, o.D[0]) : psub(o.E1, o.D[0]);
    } else {
        const V d = LIKE ? padd(o.D[B], o.D[A]) : psub(o.D[B], o.D[A]);
        return SIGN > 0 ? padd(o.E1, d) : psub(o.E1, d);
    }
}

// The node mirrored in x: its right-moving values are the mirror image's left-moving ones.  With a
// shared flux the mirrored node's B_x differs from the others, so the three left-moving values that
// the halo column sends are formed here directly.  m: +1 as it stands, -1 mirrored.
// L(x axis) = E0 + m A_x;  (x, b) like-sign plus: E1 + (D_b + m D_x);  (x, b) unlike-sign minus: E1 - (D_b - m D_x).
template <bool SHARED, typename T, int DIM>
__device__ __forceinline__ T ncde_edge_axis(const NcdeParts<One<T>, DIM>& o, bool mirrored) {
    const T a = o.A[0].v;
    return mirrored ? rsub(o.E0.v, a) : radd(o.E0.v, a);
}
template <bool SHARED, int B, bool PLUS, typename T, int DIM>
__device__ __forceinline__ T ncde_edge_diag(const NcdeParts<One<T>, DIM>& o, bool mirrored) {
    if constexpr (SHARED) {
        // D_b = D_x: the like-sign sum is D[0], the unlike one 0; mirroring swaps them
        const T d = PLUS ? (mirrored ? T(0) : o.D[0].v) : (mirrored ? o.D[0].v : T(0));
        return PLUS ? radd(o.E1.v, d) : rsub(o.E1.v, d);
    } else {
        const T x = mirrored ? -o.D[0].v : o.D[0].v;
        return PLUS ? radd(o.E1.v, radd(o.D[B].v, x)) : rsub(o.E1.v, rsub(o.D[B].v, x));
    }
}

// L(x + 1) + R(x - 1), the outer columns from the neighbouring lanes.
template <typename T>
__device__ __forceinline__ void shift_sum(const Pk<T> (&L)[2], const Pk<T> (&R)[2], Pk<T> (&s)[2]) {
    constexpr unsigned FULL = 0xffffffffu;
    const T l4 = __shfl_down_sync(FULL, L[0].lo(), 1);
    const T rm = __shfl_up_sync(FULL, R[1].hi(), 1);
    s[0] = Pk<T>::make(radd(L[0].hi(), rm), radd(L[1].lo(), R[0].lo()));
    s[1] = Pk<T>::make(radd(L[1].hi(), R[0].hi()), radd(l4, R[1].lo()));
}
// The same with the halo columns' value h in the outer columns of lanes 0 and 31.
template <typename T>
__device__ __forceinline__ void shift_sum_edge(const Pk<T> (&L)[2], const Pk<T> (&R)[2], T h, int lane, Pk<T> (&s)[2]) {
    T a[4], b[4];
    shift_lr_edge<T>(L, R, h, lane, a, b);
    sum4<T>(a, b, s);
}

}  // namespace MMFD_PK_NS
}  // namespace mmfd
