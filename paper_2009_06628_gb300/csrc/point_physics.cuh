// Pointwise Crank-Nicolson VMS physics at one quadrature point: the primal map of
// Definition 2, its tangent (J x) and its adjoint (J^T w), written out by hand.
//
// Reference ("hat") gradients.  The element map is a scaling, so a physical derivative is
// d_j = s_j D_j with D_j the derivative that the basis exchange of the element kernels leaves
// (without its scale) and s_j one number per point: on Q1 s_j = +-f/(h c_+), the sign being
// that of the thread's Gauss point along axis j and f the scale of the exchange; on Q2
// s_j = 2/h.  s_j^2 = kap is the same for every axis.  All gradients enter and all gradient
// fluxes leave in this form: instead of scaling 3 components of 7 fields and 6 fluxes, only the
// advecting vectors (v, the mass flux) carry an s_j, and the products of two gradients take kap
// from a per-level constant.  (The scale comes after the differences: nodal values scaled
// first would round before they cancel.)
//
// Mass flux.  rho v.grad v_i + (1/Pe) J.grad v_i is one product k.grad v_i with
// k = rho v + J/Pe = rho v - alpha m, m = grad mu/(Pe Cn) (J = -(alpha/Cn) grad mu), and the
// momentum row's value part with its subgrid convection is
// rho a_i + b.grad v_i, b = k - tau_m R_m; the subgrid product is S_i b_j with S = (tau_m/rho) R_m,
// which is also the solenoidality flux; g (|v|^2 + v.J/(rho Pe)) of tau_m is g (v.k)/rho.
// The map takes about 155 operations per point in 3D where the term-by-term form took 350: on the FP64 pipe, which
// bounds the FP64 kernels, that is the whole cost.
//
// S is the working type: double (one Gauss point), or float2 (two Gauss points of one element,
// packed FP32 instructions).  R_m, R_phi, tau's: Definition 2 and the strong residuals after it.
#pragma once

#include <cuda_runtime.h>

// ---- arithmetic of the working types ------------------------------------------------
__device__ __forceinline__ double fma3(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double nfma3(double a, double b, double c) { return fma(-a, b, c); }
__device__ __forceinline__ double mul2(double a, double b) { return a * b; }
__device__ __forceinline__ double add2(double a, double b) { return a + b; }
__device__ __forceinline__ double sub2(double a, double b) { return a - b; }
__device__ __forceinline__ double neg1(double a) { return -a; }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
__device__ __forceinline__ double inv_sqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ bool is_nan(double x) { return !(x == x); }

__device__ __forceinline__ float fma3(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float nfma3(float a, float b, float c) { return fmaf(-a, b, c); }
__device__ __forceinline__ float mul2(float a, float b) { return a * b; }
__device__ __forceinline__ float add2(float a, float b) { return a + b; }
__device__ __forceinline__ float sub2(float a, float b) { return a - b; }
__device__ __forceinline__ float neg1(float a) { return -a; }
__device__ __forceinline__ float recip(float x) { return 1.0f / x; }
__device__ __forceinline__ float inv_sqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ bool is_nan(float x) { return !(x == x); }

// packed FP32 (one instruction for two points)
__device__ __forceinline__ float2 fma3(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg1(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 nfma3(float2 a, float2 b, float2 c) { return __ffma2_rn(neg1(a), b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg1(b)); }
__device__ __forceinline__ float2 recip(float2 x) { return make_float2(1.0f / x.x, 1.0f / x.y); }
__device__ __forceinline__ float2 inv_sqrt(float2 x) { return make_float2(rsqrtf(x.x), rsqrtf(x.y)); }
__device__ __forceinline__ bool is_nan(float2 x) { return is_nan(x.x) || is_nan(x.y); }

// the scalar type of a working type, and a number as a working type
template <class S> struct Scalar { using type = S; };
template <> struct Scalar<float2> { using type = float; };
template <class S> __host__ __device__ __forceinline__ S splat(double a) { return S(a); }
template <> __host__ __device__ __forceinline__ float2 splat<float2>(double a) { return make_float2((float)a, (float)a); }

// Index of the mixed second derivative (i != j) in the packed array
// (2D: xy; 3D: xy, xz, yz).
__host__ __device__ __forceinline__ constexpr int hidx(int i, int j) {
    return (i < j) ? (i == 0 ? j - 1 : 2) : (j == 0 ? i - 1 : 2);
}

// Constants of one time step.
template <class S>
struct PwConst {
    S alpha, beta;       // rho = alpha phi* + beta
    S c2, c5;            // eta/Re = c2 phi* + c5
    S inv_Fr, td, c0;    // 1/Fr, 2/dt, 4/dt^2
    S inv_We;
    S gk;                // (4/h^2)/kap: a number of the basis
};
// Constants of one element level (h), built on the host in FP64.
template <class S>
struct PwLevel {
    S s;                 // |s_j|
    S kap;               // s_j^2
    S vol;               // |det J| times the scale that the exchange leaves
    S nak, km;           // -alpha kap/(Pe Cn), kap/(Pe Cn)
    S nc2k;              // -c2 kap
    S cnk;               // Cn kap
    S cn2k;              // Cn^2 kap
    S c3, c3x2;          // C_I tr(G G) / 1 and twice that
    S c0p;               // 4/dt^2 + C_phi tr(G G)/(Pe Cn)^2
    S ct;                // 1/(We tr G)
    S c4;                // C_phi tr(G G)/(Pe Cn)^2
};

// Inputs at the point: mid-point averages, D_j gradients (hats).
template <int D, class S>
struct PwIn {
    S v[D], gv[D][D], gp[D], phi, gq[D], H[D == 2 ? 1 : 3], gm[D];   // H: d_ij phi = s_i s_j H_ij
    S a[D];                       // (v^{k+1} - v^k)/dt
    S pdt;                        // (phi^{k+1} - phi^k)/dt
    S ps, gs[D];                  // phi* and its gradient
    S Hd[D], lapv[D], lapmu;      // Q2 only: pure second derivatives of phi, Laplacians of v and mu
};

// Everything the tangent and the adjoint need of the primal point.
template <int D, class S>
struct PwState {
    S vh[D], gv[D][D], phi, gq[D], H[D == 2 ? 1 : 3], a[D], gm[D];
    S rho, E, irho, er, kh[D], keh[D], qk[D], Rm[D], Rc, Rphi, vk, rad, tm, tp, tmr, Sv[D], Sh[D], bh[D], cc, EK;
    S Hl[D], lapv[D], lapmu;      // Q2 only: D_ii phi + lap phi, lap v, lap mu
};

// sg[j]: the s_j of this point (signed).
template <int D, class S, bool Q2>
__device__ __forceinline__ void pw_primal(const PwIn<D, S>& X, const PwConst<S>& c, const PwLevel<S>& L,
                                          const S sg[D], PwState<D, S>& P) {
    P.phi = X.phi;
    P.rho = fma3(c.alpha, X.ps, c.beta);
    P.E = fma3(c.c2, X.ps, c.c5);
    P.EK = mul2(P.E, L.kap);
#pragma unroll
    for (int j = 0; j < D; ++j) {
        P.vh[j] = mul2(sg[j], X.v[j]);
        P.gm[j] = X.gm[j];
        P.kh[j] = fma3(L.nak, X.gm[j], mul2(P.rho, P.vh[j]));
        P.keh[j] = fma3(L.nc2k, X.gs[j], P.kh[j]);
        P.gq[j] = X.gq[j];
        P.qk[j] = mul2(L.cnk, X.gq[j]);
        P.a[j] = X.a[j];
    }
    P.a[D - 1] = add2(X.a[D - 1], c.inv_Fr);
#pragma unroll
    for (int k = 0; k < (D == 2 ? 1 : 3); ++k) P.H[k] = X.H[k];
    S lap = splat<S>(0.0);
    if constexpr (Q2) {
#pragma unroll
        for (int j = 0; j < D; ++j) lap = add2(lap, X.Hd[j]);
        P.lapmu = X.lapmu;
    }
#pragma unroll
    for (int i = 0; i < D; ++i) {
        S ch = X.gp[i];
#pragma unroll
        for (int j = 0; j < D; ++j)
            if (j != i) ch = fma3(X.H[hidx(i, j)], P.qk[j], ch);
        if constexpr (Q2) {
            P.Hl[i] = add2(X.Hd[i], lap);
            ch = fma3(P.Hl[i], P.qk[i], ch);
        }
        S r = fma3(mul2(sg[i], c.inv_We), ch, mul2(P.rho, P.a[i]));
#pragma unroll
        for (int j = 0; j < D; ++j) {
            P.gv[i][j] = X.gv[i][j];
            r = fma3(P.keh[j], X.gv[i][j], r);
        }
        if constexpr (Q2) {
            P.lapv[i] = X.lapv[i];
            r = nfma3(P.EK, X.lapv[i], r);
        }
        P.Rm[i] = r;
    }
    P.Rc = mul2(sg[0], X.gv[0][0]);
    P.vk = mul2(P.vh[0], P.kh[0]);
    S vv = mul2(P.vh[0], P.vh[0]);
    S vq = fma3(P.vh[0], X.gq[0], X.pdt);
#pragma unroll
    for (int j = 1; j < D; ++j) {
        P.Rc = fma3(sg[j], X.gv[j][j], P.Rc);
        P.vk = fma3(P.vh[j], P.kh[j], P.vk);
        vv = fma3(P.vh[j], P.vh[j], vv);
        vq = fma3(P.vh[j], X.gq[j], vq);
    }
    P.Rphi = fma3(X.phi, P.Rc, vq);
    if constexpr (Q2) P.Rphi = nfma3(L.km, X.lapmu, P.Rphi);
    P.irho = recip(P.rho);
    P.er = mul2(P.E, P.irho);
    P.rad = fma3(c.gk, mul2(P.irho, P.vk), fma3(L.c3, mul2(P.er, P.er), c.c0));
    P.tm = inv_sqrt(P.rad);
    P.tp = inv_sqrt(fma3(c.gk, vv, L.c0p));
    P.tmr = mul2(P.tm, P.irho);
#pragma unroll
    for (int j = 0; j < D; ++j) {
        P.Sv[j] = mul2(P.tmr, P.Rm[j]);
        P.Sh[j] = mul2(sg[j], P.Sv[j]);
        P.bh[j] = nfma3(P.rho, P.Sh[j], P.kh[j]);
    }
    P.cc = fma3(P.tp, P.Rphi, neg1(P.phi));
}

// Fluxes: F0[f] multiplies N_a, F1[f][k] multiplies D_k N_a (the s_k is in F1); p: p/We.
template <int D, class S>
__device__ __forceinline__ void pw_flux(const PwState<D, S>& P, S p, S mu, S pdt, S divnew, const PwConst<S>& c,
                                        const PwLevel<S>& L, const S sg[D], S F0[D + 3], S F1[D + 3][D]) {
    const S diag = sub2(mul2(mul2(L.ct, mul2(P.tm, P.rad)), mul2(P.rho, P.Rc)), p);
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const S nq = neg1(mul2(mul2(sg[i], c.inv_We), P.qk[i]));
        S f = mul2(P.rho, P.a[i]);
#pragma unroll
        for (int j = 0; j < D; ++j) {
            f = fma3(P.bh[j], P.gv[i][j], f);
            S t = fma3(P.Sv[i], P.bh[j], fma3(nq, P.gq[j], mul2(P.EK, P.gv[i][j])));
            if (i == j) t = fma3(sg[i], diag, t);
            F1[i][j] = t;
        }
        F0[i] = f;
        F1[D][i] = P.Sh[i];
        F1[D + 1][i] = fma3(P.vh[i], P.cc, fma3(P.Sh[i], P.phi, mul2(L.km, P.gm[i])));
        F1[D + 2][i] = mul2(L.cn2k, P.gq[i]);
    }
    F0[D] = divnew;
    F0[D + 1] = pdt;
    F0[D + 2] = fma3(fma3(P.phi, P.phi, splat<S>(-1.0)), P.phi, neg1(mu));
}

// Tangent: X holds the tangents of the averages (half of the tangent of U^{k+1}; the time
// differences move by (2/dt) times those, so X.a and X.pdt are not read), dp and dmu those of
// p/We and mu.
template <int D, class S, bool Q2>
__device__ __forceinline__ void pw_tangent(const PwState<D, S>& P, const PwIn<D, S>& X, S dp, S dmu,
                                           const PwConst<S>& c, const PwLevel<S>& L, const S sg[D], S F0[D + 3],
                                           S F1[D + 3][D]) {
    const S drho = mul2(c.alpha, X.ps), dE = mul2(c.c2, X.ps);
    const S dirho = neg1(mul2(mul2(P.irho, P.irho), drho));
    const S rtd = mul2(P.rho, c.td);
    S dvh[D], dkh[D], dkeh[D], dqk[D], dbase[D], dRm[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        dvh[j] = mul2(sg[j], X.v[j]);
        dkh[j] = fma3(P.rho, dvh[j], fma3(drho, P.vh[j], mul2(L.nak, X.gm[j])));
        dkeh[j] = fma3(L.nc2k, X.gs[j], dkh[j]);
        dqk[j] = mul2(L.cnk, X.gq[j]);
        dbase[j] = fma3(rtd, X.v[j], mul2(drho, P.a[j]));
    }
    S dlap = splat<S>(0.0);
    if constexpr (Q2) {
#pragma unroll
        for (int j = 0; j < D; ++j) dlap = add2(dlap, X.Hd[j]);
    }
    const S dEK = mul2(dE, L.kap);
#pragma unroll
    for (int i = 0; i < D; ++i) {
        S ch = X.gp[i];
#pragma unroll
        for (int j = 0; j < D; ++j)
            if (j != i) ch = fma3(X.H[hidx(i, j)], P.qk[j], fma3(P.H[hidx(i, j)], dqk[j], ch));
        if constexpr (Q2) ch = fma3(add2(X.Hd[i], dlap), P.qk[i], fma3(P.Hl[i], dqk[i], ch));
        S r = fma3(mul2(sg[i], c.inv_We), ch, dbase[i]);
#pragma unroll
        for (int j = 0; j < D; ++j) r = fma3(dkeh[j], P.gv[i][j], fma3(P.keh[j], X.gv[i][j], r));
        if constexpr (Q2) r = nfma3(dEK, P.lapv[i], nfma3(P.EK, X.lapv[i], r));
        dRm[i] = r;
    }
    S dRc = mul2(sg[0], X.gv[0][0]);
    S dvk = fma3(dvh[0], P.kh[0], mul2(P.vh[0], dkh[0]));
    S vdv = mul2(P.vh[0], dvh[0]);
    S dvq = fma3(dvh[0], P.gq[0], mul2(P.vh[0], X.gq[0]));
#pragma unroll
    for (int j = 1; j < D; ++j) {
        dRc = fma3(sg[j], X.gv[j][j], dRc);
        dvk = fma3(dvh[j], P.kh[j], fma3(P.vh[j], dkh[j], dvk));
        vdv = fma3(P.vh[j], dvh[j], vdv);
        dvq = fma3(dvh[j], P.gq[j], fma3(P.vh[j], X.gq[j], dvq));
    }
    S dRphi = fma3(add2(c.td, P.Rc), X.phi, fma3(P.phi, dRc, dvq));
    if constexpr (Q2) dRphi = nfma3(L.km, X.lapmu, dRphi);
    const S der = fma3(dE, P.irho, mul2(P.E, dirho));
    const S drad = fma3(c.gk, fma3(dirho, P.vk, mul2(P.irho, dvk)), mul2(mul2(L.c3x2, P.er), der));
    const S tm2 = mul2(P.tm, P.tm), tp2 = mul2(P.tp, P.tp);
    const S dtm = mul2(mul2(splat<S>(-0.5), mul2(tm2, P.tm)), drad);
    const S dtp = neg1(mul2(mul2(c.gk, mul2(tp2, P.tp)), vdv));
    const S dtmr = fma3(dtm, P.irho, mul2(P.tm, dirho));
    const S dcc = fma3(dtp, P.Rphi, fma3(P.tp, dRphi, neg1(X.phi)));
    S dS[D], dSh[D], dbh[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        dS[j] = fma3(P.tmr, dRm[j], mul2(dtmr, P.Rm[j]));
        dSh[j] = mul2(sg[j], dS[j]);
        dbh[j] = nfma3(P.rho, dSh[j], nfma3(drho, P.Sh[j], dkh[j]));
    }
    // d(rho tau_c R_c)/We with tau_c = sqrt(rad)/tr G: d sqrt(rad) = tm drad / 2
    const S w = mul2(L.ct, P.tm);
    const S ddiag = fma3(mul2(w, P.rad), fma3(drho, P.Rc, mul2(P.rho, dRc)),
                         fma3(mul2(mul2(splat<S>(0.5), w), mul2(P.rho, P.Rc)), drad, neg1(dp)));
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const S nsg = neg1(mul2(sg[i], c.inv_We));
        const S nq = mul2(nsg, P.qk[i]), dnq = mul2(nsg, dqk[i]);
        S f = dbase[i];
#pragma unroll
        for (int j = 0; j < D; ++j) {
            f = fma3(dbh[j], P.gv[i][j], fma3(P.bh[j], X.gv[i][j], f));
            S t = fma3(P.Sv[i], dbh[j], mul2(dS[i], P.bh[j]));
            t = fma3(nq, X.gq[j], fma3(dnq, P.gq[j], t));
            t = fma3(P.EK, X.gv[i][j], fma3(dEK, P.gv[i][j], t));
            if (i == j) t = fma3(sg[i], ddiag, t);
            F1[i][j] = t;
        }
        F0[i] = f;
        F1[D][i] = dSh[i];
        F1[D + 1][i] = fma3(dvh[i], P.cc, fma3(P.vh[i], dcc, fma3(dSh[i], P.phi, fma3(P.Sh[i], X.phi, mul2(L.km, X.gm[i])))));
        F1[D + 2][i] = mul2(L.cn2k, X.gq[i]);
    }
    F0[D] = add2(dRc, dRc);
    F0[D + 1] = mul2(c.td, X.phi);
    F0[D + 2] = fma3(fma3(mul2(splat<S>(3.0), P.phi), P.phi, splat<S>(-1.0)), X.phi, neg1(dmu));
}

// Tangent for a basis function of one field alone (field F: v_F, p = D, mu = D + 2; for phi use
// pw_tangent): n its averaged value, g[k] its D_k derivatives.  The terms that such a tangent
// does not move are left out, which is more than half of them.
template <int D, class S, int F>
__device__ __forceinline__ void pw_unit(const PwState<D, S>& P, S n, const S g[D], const PwConst<S>& c,
                                        const PwLevel<S>& L, const S sg[D], S F0[D + 3], S F1[D + 3][D]) {
    const S z0 = splat<S>(0.0);
    const S w = mul2(L.ct, P.tm), tm2 = mul2(P.tm, P.tm);
    S dRm[D], dkh[D], dS[D], dSh[D], dbh[D], ddiag = z0, dtmr = z0, dcc = z0, dvh = z0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        F0[i] = z0;
        dkh[i] = z0;
        F1[D + 2][i] = z0;
    }
    F0[D] = F0[D + 1] = F0[D + 2] = z0;
    if constexpr (F < D) {
        dvh = mul2(sg[F], n);
        dkh[F] = mul2(P.rho, dvh);
        const S dbase = mul2(mul2(P.rho, c.td), n);
        const S dRc = mul2(sg[F], g[F]);
        const S drad = mul2(mul2(c.gk, P.irho), fma3(dvh, P.kh[F], mul2(P.vh[F], dkh[F])));
        const S dtp = neg1(mul2(mul2(c.gk, mul2(mul2(P.tp, P.tp), P.tp)), mul2(P.vh[F], dvh)));
        dtmr = mul2(mul2(mul2(splat<S>(-0.5), mul2(tm2, P.tm)), drad), P.irho);
        dcc = fma3(dtp, P.Rphi, mul2(P.tp, fma3(P.phi, dRc, mul2(dvh, P.gq[F]))));
        ddiag = fma3(mul2(w, P.rad), mul2(P.rho, dRc), mul2(mul2(mul2(splat<S>(0.5), w), mul2(P.rho, P.Rc)), drad));
        S r = dbase, f = dbase;
#pragma unroll
        for (int j = 0; j < D; ++j) {
            r = fma3(P.keh[j], g[j], r);
            f = fma3(P.bh[j], g[j], f);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) dRm[i] = i == F ? fma3(dkh[F], P.gv[i][F], r) : mul2(dkh[F], P.gv[i][F]);
        F0[F] = f;
        F0[D] = add2(dRc, dRc);
    } else if constexpr (F == D) {
#pragma unroll
        for (int i = 0; i < D; ++i) dRm[i] = mul2(mul2(sg[i], c.inv_We), g[i]);
        ddiag = neg1(mul2(c.inv_We, n));
    } else {
        S dvk = z0;
#pragma unroll
        for (int j = 0; j < D; ++j) {
            dkh[j] = mul2(L.nak, g[j]);
            dvk = fma3(P.vh[j], dkh[j], dvk);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            S r = z0;
#pragma unroll
            for (int j = 0; j < D; ++j) r = fma3(dkh[j], P.gv[i][j], r);
            dRm[i] = r;
        }
        const S drad = mul2(mul2(c.gk, P.irho), dvk);
        dtmr = mul2(mul2(mul2(splat<S>(-0.5), mul2(tm2, P.tm)), drad), P.irho);
        ddiag = mul2(mul2(mul2(splat<S>(0.5), w), mul2(P.rho, P.Rc)), drad);
        F0[D + 2] = neg1(n);
    }
#pragma unroll
    for (int j = 0; j < D; ++j) {
        dS[j] = F == D ? mul2(P.tmr, dRm[j]) : fma3(P.tmr, dRm[j], mul2(dtmr, P.Rm[j]));
        dSh[j] = mul2(sg[j], dS[j]);
        dbh[j] = nfma3(P.rho, dSh[j], dkh[j]);
    }
#pragma unroll
    for (int i = 0; i < D; ++i) {
#pragma unroll
        for (int j = 0; j < D; ++j) {
            F0[i] = fma3(dbh[j], P.gv[i][j], F0[i]);
            S t = fma3(P.Sv[i], dbh[j], mul2(dS[i], P.bh[j]));
            if (F < D && i == F) t = fma3(P.EK, g[j], t);
            if (i == j) t = fma3(sg[i], ddiag, t);
            F1[i][j] = t;
        }
        F1[D][i] = dSh[i];
        S t = mul2(dSh[i], P.phi);
        if (F < D) t = fma3(P.vh[i], dcc, t);
        if (F < D && i == F) t = fma3(dvh, P.cc, t);
        if (F == D + 2) t = fma3(L.km, g[i], t);
        F1[D + 1][i] = t;
    }
}

// Adjoint: F0, F1 hold the cotangents of the fluxes (value and D_k gradient of the test field);
// returns the cotangents of the inputs in Xb (Xb.a, Xb.pdt those of the time differences), of
// p/We, mu and div v^{k+1}, and of Cn.  iCn = 1/Cn.
template <int D, class S, bool Q2>
__device__ __forceinline__ void pw_adjoint(const PwState<D, S>& P, const S F0[D + 3], const S F1[D + 3][D],
                                           const PwConst<S>& c, const PwLevel<S>& L, const S sg[D], S iCn,
                                           PwIn<D, S>& Xb, S& pb, S& mub, S& divb, S& Cnb) {
    const S z0 = splat<S>(0.0);
    S diagb = z0, EKb = z0, cb = z0, Sb[D], bhb[D], Shb[D], vhb[D], khb[D], qkb[D], rhob = z0;
    S phib, Rcb, irhob, Eb, radb;
    Cnb = z0;
#pragma unroll
    for (int j = 0; j < D; ++j) bhb[j] = z0;
#pragma unroll
    for (int j = 0; j < D; ++j) Xb.gq[j] = mul2(L.cn2k, F1[D + 2][j]);
#pragma unroll
    for (int j = 0; j < D; ++j) Cnb = fma3(P.gq[j], Xb.gq[j], Cnb);      // Cn^2: twice, below
    Cnb = add2(Cnb, Cnb);
    const S z = F0[D + 2];
    phib = mul2(fma3(mul2(splat<S>(3.0), P.phi), P.phi, splat<S>(-1.0)), z);
    mub = neg1(z);
#pragma unroll
    for (int i = 0; i < D; ++i) {
        diagb = fma3(sg[i], F1[i][i], diagb);
        S sb = z0, nqb = z0;
        const S nsw = neg1(mul2(sg[i], c.inv_We)), nq = mul2(nsw, P.qk[i]);
#pragma unroll
        for (int j = 0; j < D; ++j) {
            const S fb = F1[i][j];
            sb = fma3(P.bh[j], fb, sb);
            nqb = fma3(P.gq[j], fb, nqb);
            bhb[j] = fma3(P.Sv[i], fb, fma3(P.gv[i][j], F0[i], bhb[j]));
            Xb.gq[j] = fma3(nq, fb, Xb.gq[j]);
            EKb = fma3(P.gv[i][j], fb, EKb);
            Xb.gv[i][j] = fma3(P.EK, fb, mul2(P.bh[j], F0[i]));
        }
        Sb[i] = sb;
        qkb[i] = mul2(nsw, nqb);
        const S y = F1[D + 1][i];
        vhb[i] = mul2(P.cc, y);
        cb = fma3(P.vh[i], y, cb);
        Shb[i] = fma3(P.phi, y, F1[D][i]);
        phib = fma3(P.Sh[i], y, phib);
        Xb.gm[i] = mul2(L.km, y);
    }
    divb = F0[D];
    pb = neg1(diagb);
    {
        const S w = mul2(L.ct, P.tm), x = mul2(mul2(w, P.rad), diagb);
        radb = mul2(mul2(mul2(splat<S>(0.5), w), mul2(P.rho, P.Rc)), diagb);
        rhob = mul2(P.Rc, x);
        Rcb = mul2(P.rho, x);
    }
    const S Rphib = mul2(P.tp, cb);
    phib = sub2(phib, cb);
    {
        const S tp3 = mul2(mul2(P.tp, P.tp), P.tp);
        const S radpb = mul2(mul2(splat<S>(-0.5), tp3), mul2(P.Rphi, cb));
        const S two_vvb = mul2(add2(c.gk, c.gk), radpb);
        Cnb = nfma3(mul2(splat<S>(2.0), L.c4), radpb, Cnb);
#pragma unroll
        for (int j = 0; j < D; ++j) vhb[j] = fma3(P.vh[j], two_vvb, fma3(P.gq[j], Rphib, vhb[j]));
    }
    S tmrb = z0;
    S Rmb[D], kehb[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        khb[j] = bhb[j];
        Shb[j] = nfma3(P.rho, bhb[j], Shb[j]);
        rhob = nfma3(P.Sh[j], bhb[j], rhob);
        const S sb = fma3(sg[j], Shb[j], Sb[j]);
        Rmb[j] = mul2(P.tmr, sb);
        tmrb = fma3(P.Rm[j], sb, tmrb);
        kehb[j] = z0;
    }
    irhob = mul2(P.tm, tmrb);
    {
        const S tm3 = mul2(mul2(P.tm, P.tm), P.tm);
        radb = fma3(mul2(splat<S>(-0.5), tm3), mul2(P.irho, tmrb), radb);
    }
    const S gr = mul2(c.gk, radb);
    const S vkb = mul2(gr, P.irho);
    irhob = fma3(gr, P.vk, irhob);
    const S erb = mul2(mul2(L.c3x2, P.er), radb);
    irhob = fma3(P.E, erb, irhob);
    phib = fma3(P.Rc, Rphib, phib);
    Rcb = fma3(P.phi, Rphib, Rcb);
    Xb.pdt = add2(F0[D + 1], Rphib);
    if constexpr (Q2) {
        Xb.lapmu = neg1(mul2(L.km, Rphib));
        Cnb = nfma3(P.lapmu, Xb.lapmu, Cnb);
    }
    S lapb = z0;
#pragma unroll
    for (int k = 0; k < (D == 2 ? 1 : 3); ++k) Xb.H[k] = z0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const S rb = Rmb[i], bb = add2(F0[i], rb), ch = mul2(mul2(sg[i], c.inv_We), rb);
        rhob = fma3(P.a[i], bb, rhob);
        Xb.a[i] = mul2(P.rho, bb);
        Xb.gp[i] = ch;
#pragma unroll
        for (int j = 0; j < D; ++j) {
            kehb[j] = fma3(P.gv[i][j], rb, kehb[j]);
            Xb.gv[i][j] = fma3(P.keh[j], rb, Xb.gv[i][j]);
            if (j != i) {
                Xb.H[hidx(i, j)] = fma3(P.qk[j], ch, Xb.H[hidx(i, j)]);
                qkb[j] = fma3(P.H[hidx(i, j)], ch, qkb[j]);
            }
        }
        Xb.gv[i][i] = fma3(sg[i], Rcb, Xb.gv[i][i]);
        if constexpr (Q2) {
            EKb = nfma3(P.lapv[i], rb, EKb);
            Xb.lapv[i] = neg1(mul2(P.EK, rb));
            qkb[i] = fma3(P.Hl[i], ch, qkb[i]);
            Xb.Hd[i] = mul2(P.qk[i], ch);
            lapb = add2(lapb, Xb.Hd[i]);
        }
    }
    Eb = fma3(L.kap, EKb, mul2(P.irho, erb));
#pragma unroll
    for (int j = 0; j < D; ++j) {
        if constexpr (Q2) Xb.Hd[j] = add2(Xb.Hd[j], lapb);
        Cnb = fma3(P.qk[j], qkb[j], Cnb);
        Xb.gq[j] = fma3(L.cnk, qkb[j], fma3(P.vh[j], Rphib, Xb.gq[j]));
        Xb.gs[j] = mul2(L.nc2k, kehb[j]);
        const S kb = fma3(P.vh[j], vkb, add2(khb[j], kehb[j]));
        vhb[j] = fma3(P.kh[j], vkb, fma3(P.rho, kb, vhb[j]));
        rhob = fma3(P.vh[j], kb, rhob);
        Xb.gm[j] = fma3(L.nak, kb, Xb.gm[j]);
        Cnb = nfma3(P.gm[j], Xb.gm[j], Cnb);
        Xb.v[j] = mul2(sg[j], vhb[j]);
    }
    rhob = nfma3(mul2(P.irho, P.irho), irhob, rhob);
    Xb.phi = phib;
    Xb.ps = fma3(c.alpha, rhob, mul2(c.c2, Eb));
    Cnb = mul2(Cnb, iCn);
}
