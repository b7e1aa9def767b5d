// nse_class.cuh -- the lean He-Luo NSE step in class form, on pairs of neighbouring nodes.
//
// With streaming momentum (Coef::nA) a node sends one value v_j = E_p +- O_p along each direction
// j, and an output node's moments are
//     rho' = c rho-part + sum_j v_j,   u_a' = nsm (sum over e_ja = +-1 of -+ v_j) + ab0 u_a,
// so each value has to be added once per moment it enters, whatever the node it came from.  The
// values are therefore grouped by the direction's class along each axis and summed within a class
// before the classes are combined:
//   - along x, the values moving left (L, they come from column x + 1) and right (R, from x - 1)
//     are needed as their sum (rho and the other momenta) and difference (u_x);
//   - along the marching axis, the whole group that an input row (plane) sends to the row behind
//     (P), to its own (C) or to the one ahead (N) enters that axis's momentum with one sign.
// Against pushing each v_j into every accumulator (lean_push_sv) that is 42 instead of 58
// floating-point operations per D2Q9 node and step, no node is evaluated twice (the x neighbours'
// sums come from the neighbouring lanes), and, the main gain, every operation but the six x-shifted
// sums acts on the lane's columns (0, 1) and (2, 3) alike: FP32 runs them as paired instructions
// (fma.f32x2 and the like), which halves the issue slots the step was bound by.
#pragma once

#include "pk.cuh"
#include "stencil.cuh"

namespace mmfd {
inline namespace MMFD_PK_NS {


// The class form's coefficients of one level, from Coef (axis pairs: index 0, diagonal pairs: the
// first diagonal pair; the host checks that a class shares them).
template <typename T>
struct ClassCoef {
    Pk<T> nA[2], nU[2], nk[2], no[2], mo[2];   // k: 0 axis pairs, 1 diagonal pairs; mo = -no
    Pk<T> nc[2];                               // rest: a0 rho + a+ f_0^eq = nc[0] rho + nc[1] |u|^2
    Pk<T> nsm, msm;                            // kappa c / rho0, and minus that
    Pk<T> ab0;
};

// ab0 as the class forms take it: a uniform velocity comes out of one step times ab0 + k, k the sum of the
// rounded odd coefficients, which should be umom; in FP32 ab0 takes up what their rounding left (LBGK at
// d_0 = 1/3 drifted by 2e-8 a step without).
template <typename T>
T class_ab0(T ab0, double k, double umom) {
    return sizeof(T) == 8 ? ab0 : (T)(umom - k);
}

template <int LAT, typename T>
ClassCoef<T> class_coef(const Coef<T>& cf, double umom, int l) {
    constexpr int DG = lat_dim(LAT);   // first diagonal pair
    ClassCoef<T> c;
    for (int k = 0; k < 2; ++k) {
        c.nA[k] = Pk<T>::fill(cf.nA[l][k]);
        c.nU[k] = Pk<T>::fill(cf.nU[l][k]);
        c.nk[k] = Pk<T>::fill(cf.nk[l][k == 0 ? 0 : DG]);
        c.no[k] = Pk<T>::fill(cf.no[l][k == 0 ? 0 : DG]);
        c.mo[k] = Pk<T>::fill(-cf.no[l][k == 0 ? 0 : DG]);
        c.nc[k] = Pk<T>::fill(cf.nc[l][k]);
    }
    c.nsm = Pk<T>::fill(cf.nsm[l][0]);
    c.msm = Pk<T>::fill(-cf.nsm[l][0]);
    c.ab0 = Pk<T>::fill(class_ab0(cf.ab0[l], (double)cf.nsm[l][0] * (2.0 * cf.no[l][0] + 4.0 * (DG - 1) * cf.no[l][DG]), umom));
    return c;
}

// The same with the classes' common factors taken out, as D3Q19 with d_0 = 1/3 allows (the host checks
// it): E_p +- O_p = nA_k [ (rho + dU |u|^2) + gk (e_p . u)^2 +- be (e_p . u) ] with nA_1 = lam nA_0, so the
// diagonal classes' sums take lam once and the results nA_0.
template <typename T>
struct ClassNorm {
    T dU, gk, be, lam;
    T cR, cU;      // rest: (a0 rho + a+ f_0^eq) / nA_0 = cR rho + cU |u|^2
    T fR, fM, fD;  // nA_0, nsm nA_0, nsm nA_1
    T ab0;
};

template <typename T>
ClassNorm<T> class_norm(const Coef<T>& cf, double umom, int l) {
    ClassNorm<T> c;
    const T n0 = cf.nA[l][0];
    c.dU = cf.nU[l][0] / n0;
    c.gk = cf.nk[l][0] / n0;
    c.be = cf.no[l][0] / n0;
    c.lam = cf.nA[l][1] / n0;
    c.cR = cf.nc[l][0] / n0;
    c.cU = cf.nc[l][1] / n0;
    c.fR = n0;
    c.fM = cf.nsm[l][0] * n0;
    c.fD = cf.nsm[l][0] * cf.nA[l][1];
    c.ab0 = class_ab0(cf.ab0[l], (double)c.fM * c.be * (2.0 + 6.0 * c.lam) + 2.0 * c.fD * c.be, umom);
    return c;
}

// One row of a lane's four columns as two pairs, per field.
template <typename T, int NF>
struct RowPk {
    Pk<T> f[NF][2];
};

// The class values moving left and right, shifted to the columns they land on and combined:
// s = L(x + 1) + R(x - 1), d = L(x + 1) - R(x - 1).  The outer columns' neighbours come from the
// neighbouring lanes (lanes 0 and 31 get their own values instead: their outer column is wrong).
template <typename T>
__device__ __forceinline__ void shift_lr(const Pk<T> (&L)[2], const Pk<T> (&R)[2], Pk<T> (&s)[2], Pk<T> (&d)[2]) {
    constexpr unsigned FULL = 0xffffffffu;
    const T l4 = __shfl_down_sync(FULL, L[0].lo(), 1);
    const T rm = __shfl_up_sync(FULL, R[1].hi(), 1);
    const T a[4] = {L[0].hi(), L[1].lo(), L[1].hi(), l4};
    const T b[4] = {rm, R[0].lo(), R[0].hi(), R[1].lo()};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        s[h] = Pk<T>::make(radd(a[2 * h], b[2 * h]), radd(a[2 * h + 1], b[2 * h + 1]));
        d[h] = Pk<T>::make(rsub(a[2 * h], b[2 * h]), rsub(a[2 * h + 1], b[2 * h + 1]));
    }
}

// ------------------------------------------------------------------ D2Q9, rows marched in y

// Sums of the output rows around the current input row r: row r (it has had row r-1's N group and
// its own C group; row r+1's P group completes it) and row r+1 (row r's N group only).
template <typename T>
struct Row2 {
    Pk<T> rho[2], mx[2], my[2];   // after the C group
    Pk<T> ns[2], nd[2];           // N group: its sum and its L - R difference
};

template <typename T>
__device__ __forceinline__ void row2_clear(Row2<T>& a) {
#pragma unroll
    for (int h = 0; h < 2; ++h) a.rho[h] = a.mx[h] = a.my[h] = a.ns[h] = a.nd[h] = Pk<T>::fill(T(0));
}

// Take input row r (rho, u_x, u_y), advance the sums, and replace `in` by the completed output
// row r - 1.
template <typename T>
__device__ __forceinline__ void class_row2d(const ClassCoef<T>& c, RowPk<T, 3>& in, Row2<T>& acc) {
    using P = Pk<T>;
    P pL[2], pR[2], pE[2], cL[2], cR[2], nL[2], nR[2], nE[2], ctr[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const P rho = in.f[0][h], ux = in.f[1][h], uy = in.f[2][h];
        const P xx = pmul(ux, ux), yy = pmul(uy, uy);
        const P U = padd(xx, yy);
        const P b0 = pfma(c.nU[0], U, pmul(c.nA[0], rho));
        const P b1 = pfma(c.nU[1], U, pmul(c.nA[1], rho));
        const P e0 = pfma(c.nk[0], xx, b0), e1 = pfma(c.nk[0], yy, b0);
        const P c2 = padd(uy, ux), c3 = psub(uy, ux);
        const P e2 = pfma(c.nk[1], pmul(c2, c2), b1), e3 = pfma(c.nk[1], pmul(c3, c3), b1);
        const P o0 = c.no[0], m0 = c.mo[0], o1 = c.no[1], m1 = c.mo[1];
        cL[h] = pfma(o0, ux, e0);
        cR[h] = pfma(m0, ux, e0);
        pE[h] = pfma(o0, uy, e1);
        nE[h] = pfma(m0, uy, e1);
        pL[h] = pfma(o1, c2, e2);
        nR[h] = pfma(m1, c2, e2);
        pR[h] = pfma(o1, c3, e3);
        nL[h] = pfma(m1, c3, e3);
        ctr[h] = pfma(c.nc[1], U, pmul(c.nc[0], rho));
    }
    P s[2], d[2];
    P out[3][2];
    shift_lr<T>(pL, pR, s, d);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const P sum = padd(s[h], pE[h]);
        out[0][h] = padd(acc.rho[h], sum);
        out[1][h] = pfma(c.nsm, d[h], acc.mx[h]);
        out[2][h] = pfma(c.nsm, sum, acc.my[h]);
    }
    shift_lr<T>(cL, cR, s, d);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        acc.rho[h] = padd(padd(ctr[h], acc.ns[h]), s[h]);
        // (nsm and ab0 as they are: momentum sums kept in units of nsm take ab0 / nsm, whose rounding comes on
        // top of nsm's, and with it a uniform flow drifted up to four times as fast)
        acc.mx[h] = pfma(c.nsm, padd(acc.nd[h], d[h]), pmul(c.ab0, in.f[1][h]));
        acc.my[h] = pfma(c.msm, acc.ns[h], pmul(c.ab0, in.f[2][h]));
    }
    shift_lr<T>(nL, nR, s, d);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        acc.ns[h] = padd(s[h], nE[h]);
        acc.nd[h] = d[h];
#pragma unroll
        for (int f = 0; f < 3; ++f) in.f[f][h] = out[f][h];
    }
}

// ------------------------------------------------------------------ D3Q19, planes marched in z

// The same shift with the outer neighbours' class values given: h is the L value of the column
// right of the lane's four in lane 31 and the R value of the column left of them in lane 0.
template <typename T>
__device__ __forceinline__ void shift_lr_edge(const Pk<T> (&L)[2], const Pk<T> (&R)[2], T h, int lane, T (&a)[4], T (&b)[4]) {
    constexpr unsigned FULL = 0xffffffffu;
    const T l4 = __shfl_down_sync(FULL, L[0].lo(), 1);
    const T rm = __shfl_up_sync(FULL, R[1].hi(), 1);
    a[0] = L[0].hi(); a[1] = L[1].lo(); a[2] = L[1].hi(); a[3] = lane == 31 ? h : l4;
    b[0] = lane == 0 ? h : rm; b[1] = R[0].lo(); b[2] = R[0].hi(); b[3] = R[1].lo();
}
template <typename T>
__device__ __forceinline__ void sum4(const T (&a)[4], const T (&b)[4], Pk<T> (&s)[2]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) s[h] = Pk<T>::make(radd(a[2 * h], b[2 * h]), radd(a[2 * h + 1], b[2 * h + 1]));
}
template <typename T>
__device__ __forceinline__ void diff4(const T (&a)[4], const T (&b)[4], Pk<T> (&d)[2]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) d[h] = Pk<T>::make(rsub(a[2 * h], b[2 * h]), rsub(a[2 * h + 1], b[2 * h + 1]));
}

// Sums of one output row in the output planes around the current input plane z: plane z (it has
// had plane z-1's N group and its own C group; plane z+1's P group completes it) and plane z+1
// (plane z's N group only): the momenta as they are, rho and the N group in units of nA_0.  nx, ny are the N
// group's x and y momentum in units of nA_1; its z momentum is minus its sum.
template <typename T>
struct Row3 {
    Pk<T> rho[2], mx[2], my[2], mz[2];
    Pk<T> ns[2], nx[2], ny[2];
};

template <typename T>
__device__ __forceinline__ void row3_clear(Row3<T>& a) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
        a.rho[h] = a.mx[h] = a.my[h] = a.mz[h] = a.ns[h] = a.nx[h] = a.ny[h] = Pk<T>::fill(T(0));
}

// What the rows above and below send into an output row, combined over the two, for the lane's two
// pairs: sums (s) and differences above - below (d) of the (y, z) diagonals of the P and N groups,
// of the y axis (E), and of the (x, y) diagonals moving left (L) and right (R).
template <typename T>
struct Sides3 {
    Pk<T> sP[2], dP[2], sN[2], dN[2], sE[2], dE[2], sL[2], sR[2], dL[2], dR[2];
    T hs, hd;   // edge column: sum and difference of its (x, y) diagonal
};

// From the row above (up; its values moving to y - 1) and the row below (dn; moving to y + 1).  ue,
// de: the edge column's nodes of the two rows (rho, u; lane 0's with u_x negated, so that its
// right-moving values are the mirror image's left-moving ones, operation by operation).
template <typename T>
__device__ __forceinline__ void class_sides3d(const ClassNorm<T>& c, const RowPk<T, 4>& up, const RowPk<T, 4>& dn,
                                              const T (&ue)[4], const T (&de)[4], Sides3<T>& o) {
    using P = Pk<T>;
    const P gk = P::fill(c.gk);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        P v[2][5];   // [above, below][L, R, E, P, N]
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const RowPk<T, 4>& in = q == 0 ? up : dn;
            const P rho = in.f[0][h], ux = in.f[1][h], uy = in.f[2][h], uz = in.f[3][h];
            const P yy = pmul(uy, uy);
            const P r = pfma(P::fill(c.dU), padd(padd(pmul(ux, ux), yy), pmul(uz, uz)), rho);
            const P c3 = padd(uy, ux), c4 = psub(uy, ux), c7 = padd(uz, uy), c8 = psub(uz, uy);
            const P e3 = pfma(gk, pmul(c3, c3), r), e4 = pfma(gk, pmul(c4, c4), r);
            const P e7 = pfma(gk, pmul(c7, c7), r), e8 = pfma(gk, pmul(c8, c8), r);
            const P o = P::fill(q == 0 ? c.be : -c.be), m = P::fill(q == 0 ? -c.be : c.be);
            v[q][2] = pfma(o, uy, pfma(gk, yy, r));
            v[q][q == 0 ? 0 : 1] = pfma(o, c3, e3);
            v[q][q == 0 ? 1 : 0] = pfma(o, c4, e4);
            v[q][q == 0 ? 3 : 4] = pfma(o, c7, e7);
            v[q][q == 0 ? 4 : 3] = pfma(m, c8, e8);
        }
        o.sL[h] = padd(v[0][0], v[1][0]);
        o.dL[h] = psub(v[0][0], v[1][0]);
        o.sR[h] = padd(v[0][1], v[1][1]);
        o.dR[h] = psub(v[0][1], v[1][1]);
        o.sE[h] = padd(v[0][2], v[1][2]);
        o.dE[h] = psub(v[0][2], v[1][2]);
        o.sP[h] = padd(v[0][3], v[1][3]);
        o.dP[h] = psub(v[0][3], v[1][3]);
        o.sN[h] = padd(v[0][4], v[1][4]);
        o.dN[h] = psub(v[0][4], v[1][4]);
    }
    T h[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const T(&e)[4] = q == 0 ? ue : de;
        const T r = rfma(c.dU, radd(radd(rmul(e[1], e[1]), rmul(e[2], e[2])), rmul(e[3], e[3])), e[0]);
        const T cu = q == 0 ? radd(e[2], e[1]) : rsub(e[2], e[1]);
        h[q] = rfma(q == 0 ? c.be : -c.be, cu, rfma(c.gk, rmul(cu, cu), r));
    }
    o.hs = radd(h[0], h[1]);
    o.hd = rsub(h[0], h[1]);
}

// One output row's sums advanced by an input plane: from the row's own input nodes (in; e: its edge
// column's node) and from the rows beside it (sd).  in: replaced by the completed row of the plane
// behind.
template <typename T>
__device__ __forceinline__ void class_row3d(const ClassNorm<T>& c, RowPk<T, 4>& in, const T (&e)[4], const Sides3<T>& sd,
                                            int lane, Row3<T>& acc) {
    using P = Pk<T>;
    const P gk = P::fill(c.gk), o = P::fill(c.be), m = P::fill(-c.be), lam = P::fill(c.lam), ab0 = P::fill(c.ab0);
    const P fM = P::fill(c.fM), mM = P::fill(-c.fM), fD = P::fill(c.fD);
    P cL[2], cR[2], pL[2], pR[2], pE[2], nL[2], nR[2], nE[2], ctr[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const P rho = in.f[0][h], ux = in.f[1][h], uy = in.f[2][h], uz = in.f[3][h];
        const P xx = pmul(ux, ux), zz = pmul(uz, uz);
        const P U = padd(padd(xx, pmul(uy, uy)), zz);
        const P r = pfma(P::fill(c.dU), U, rho);
        const P e0 = pfma(gk, xx, r), e2 = pfma(gk, zz, r);
        cL[h] = pfma(o, ux, e0);
        cR[h] = pfma(m, ux, e0);
        pE[h] = pfma(o, uz, e2);
        nE[h] = pfma(m, uz, e2);
        const P c5 = padd(uz, ux), c6 = psub(uz, ux);
        const P e5 = pfma(gk, pmul(c5, c5), r), e6 = pfma(gk, pmul(c6, c6), r);
        pL[h] = pfma(o, c5, e5);
        nR[h] = pfma(m, c5, e5);
        pR[h] = pfma(o, c6, e6);
        nL[h] = pfma(m, c6, e6);
        ctr[h] = pfma(P::fill(c.cU), U, pmul(P::fill(c.cR), rho));
    }
    T hC, hP, hN;
    {
        const T xx = rmul(e[1], e[1]);
        const T r = rfma(c.dU, radd(radd(xx, rmul(e[2], e[2])), rmul(e[3], e[3])), e[0]);
        const T c5 = radd(e[3], e[1]), c6 = rsub(e[3], e[1]);
        hC = rfma(c.be, e[1], rfma(c.gk, xx, r));
        hP = rfma(c.be, c5, rfma(c.gk, rmul(c5, c5), r));
        hN = rfma(-c.be, c6, rfma(c.gk, rmul(c6, c6), r));
    }
    T a[4], b[4];
    P s[2], d[2], y[2], out[4][2];
    shift_lr_edge<T>(pL, pR, hP, lane, a, b);
    sum4<T>(a, b, s);
    diff4<T>(a, b, d);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const P sum = pfma(lam, padd(s[h], sd.sP[h]), pE[h]);
        out[0][h] = pmul(P::fill(c.fR), padd(acc.rho[h], sum));
        out[1][h] = pfma(fD, d[h], acc.mx[h]);
        out[2][h] = pfma(fD, sd.dP[h], acc.my[h]);
        out[3][h] = pfma(fM, sum, acc.mz[h]);
    }
    shift_lr_edge<T>(sd.dL, sd.dR, sd.hd, lane, a, b);
    sum4<T>(a, b, y);
    P L[2], R[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        L[h] = pfma(lam, sd.sL[h], cL[h]);
        R[h] = pfma(lam, sd.sR[h], cR[h]);
    }
    shift_lr_edge<T>(L, R, rfma(c.lam, sd.hs, hC), lane, a, b);
    sum4<T>(a, b, s);
    diff4<T>(a, b, d);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        acc.rho[h] = padd(padd(ctr[h], acc.ns[h]), padd(s[h], sd.sE[h]));
        acc.mx[h] = pfma(fM, pfma(lam, acc.nx[h], d[h]), pmul(ab0, in.f[1][h]));
        acc.my[h] = pfma(fM, pfma(lam, padd(acc.ny[h], y[h]), sd.dE[h]), pmul(ab0, in.f[2][h]));
        acc.mz[h] = pfma(mM, acc.ns[h], pmul(ab0, in.f[3][h]));
    }
    shift_lr_edge<T>(nL, nR, hN, lane, a, b);
    sum4<T>(a, b, s);
    diff4<T>(a, b, d);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        acc.ns[h] = pfma(lam, padd(s[h], sd.sN[h]), nE[h]);
        acc.nx[h] = d[h];
        acc.ny[h] = sd.dN[h];
#pragma unroll
        for (int f = 0; f < 4; ++f) in.f[f][h] = out[f][h];
    }
}

}  // namespace MMFD_PK_NS
}  // namespace mmfd
