// Triquadratic (Q2) elements (the paper's manufactured-solution study, Section 5.1, uses quadratic
// elements): residual, J x (FP64 / FP32) and J^T w of Definition 2 on uniform octrees (no hanging
// nodes), with 3^d nodes per element and the 3-point Gauss rule per axis.
//
// Lanes: 27 of a warp hold one 3D element or three 2D ones, lane i_0 + 3 i_1 (+ 9 i_2) its node and
// its Gauss point of that index; in FP32 every lane holds the same point of two elements in packed
// arithmetic.  Interpolation goes one axis at a time between the three lanes of a line (two
// shuffles, three multiply-adds for a value, a derivative or a second derivative): 27 operations
// per point for value and gradient of a field, where summing 27 basis products costs 108 and their
// evaluation as much again.  The test contraction runs the transposes with the quadrature weights
// in their coefficients.  Unlike Q1, the pure second derivatives do not vanish: the strong
// residuals take the full Hessian of phi and the Laplacians of v and mu (pw_*<..., Q2 = true>).
//   32^3 elements, FP32 J x: 303 -> 94 us; FP64 J x 10.2 -> 2.04 ms, residual 7.8 -> 1.26 ms,
//   J^T w 11.2 -> 2.31 ms.
// Bound: FP64 pipe (FP64), shuffles and FMA issue in equal parts (FP32).
#include <cuda_runtime.h>

#include <type_traits>

#include "chns_internal.h"
#include "point_physics.cuh"
#include "replaced_rows.cuh"

namespace {

template <int D>
struct Q2S {
    static constexpr int NN = D == 2 ? 9 : 27;    // nodes = Gauss points per element
    static constexpr int NF = D + 3;
    static constexpr int EPW = D == 2 ? 3 : 1;    // elements per warp (times the halves of a lane)
};
template <class S> struct Halves { static constexpr int n = 1; };
template <> struct Halves<float2> { static constexpr int n = 2; };
constexpr int Q2_THREADS = 128;

__device__ __forceinline__ double shfl(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }
__device__ __forceinline__ float2 shfl(float2 v, int l) {
    return make_float2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
__device__ __forceinline__ double pack(const double* a) { return a[0]; }
__device__ __forceinline__ float2 pack(const float* a) { return make_float2(a[0], a[1]); }
__device__ __forceinline__ double half_of(double v, int) { return v; }
__device__ __forceinline__ float half_of(float2 v, int i) { return i == 0 ? v.x : v.y; }

// 1D quadratic Lagrange polynomials L_0 = t (t - 1)/2, L_1 = 1 - t^2, L_2 = t (t + 1)/2 at the Gauss
// points t = 0, +-sqrt(3/5), their derivatives, and the weights 8/9, 5/9
constexpr double Q2_G = 0.77459666924148337704;
__device__ __forceinline__ double gp(int q) { return q == 1 ? 0.0 : (q == 0 ? -Q2_G : Q2_G); }
__device__ __forceinline__ double gw(int q) { return q == 1 ? 0.88888888888888888889 : 0.55555555555555555556; }
__device__ __forceinline__ double lag(int a, int q) {   // t^2 = 3/5 off the centre
    if (q == 1) return a == 1 ? 1.0 : 0.0;
    if (a == 1) return 0.4;
    return (a == 0) == (q == 0) ? 0.3 + 0.5 * Q2_G : 0.3 - 0.5 * Q2_G;
}
__device__ __forceinline__ double dlag(int a, int q) {
    return a == 1 ? -2.0 * gp(q) : (a == 0 ? gp(q) - 0.5 : gp(q) + 0.5);
}
// the other two lanes of this lane's line along an axis, and the coefficients of the line's values
// in the order own, n1, n2: L for a value, D for a derivative
template <class S>
struct Line {
    int d, n1, n2;       // own digit, lanes of digits d + 1 and d + 2 (mod 3)
    S L[3], D[3];
};
// TR: transposed (this lane's node, weighted by the Gauss weights of the line's points)
template <bool TR, class S>
__device__ __forceinline__ Line<S> line(int lane, int idx, int stride, bool active) {
    Line<S> l;
    l.d = active ? (idx / stride) % 3 : 0;
    const int d1 = (l.d + 1) % 3, d2 = (l.d + 2) % 3;
    l.n1 = active ? lane + (d1 - l.d) * stride : lane;
    l.n2 = active ? lane + (d2 - l.d) * stride : lane;
    const int o[3] = {l.d, d1, d2};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        l.L[i] = splat<S>(TR ? lag(l.d, o[i]) * gw(o[i]) : lag(o[i], l.d));
        l.D[i] = splat<S>(TR ? dlag(l.d, o[i]) * gw(o[i]) : dlag(o[i], l.d));
    }
    return l;
}
template <class S>
struct Tri {
    S o, p, q;
    __device__ __forceinline__ Tri(S u, const Line<S>& l) : o(u), p(shfl(u, l.n1)), q(shfl(u, l.n2)) {}
    __device__ __forceinline__ S val(const Line<S>& l) const { return fma3(l.L[2], q, fma3(l.L[1], p, mul2(l.L[0], o))); }
    __device__ __forceinline__ S der(const Line<S>& l) const { return fma3(l.D[2], q, fma3(l.D[1], p, mul2(l.D[0], o))); }
    __device__ __forceinline__ S val(const Line<S>& l, S c) const { return fma3(l.L[2], q, fma3(l.L[1], p, fma3(l.L[0], o, c))); }
    __device__ __forceinline__ S der(const Line<S>& l, S c) const { return fma3(l.D[2], q, fma3(l.D[1], p, fma3(l.D[0], o, c))); }
};
// The same from the differences to the own value, for values and derivatives of nodal data together (no more
// operations: L sums to 1 and D to 0 over a line).  A derivative as a sum of products rounds at the size of
// the data, which in the phases is 1 where the derivative is 0; so it rounds at the size of the variation.
//   Against 64 bits, 2D 32^2: solenoidality row of the residual 6.1e-15 -> 3.4e-15, potential row 7.9e-15 ->
//   5.5e-15, all rows 9.6e-16 -> 8.1e-16, FP32 J x 1.0e-7 -> 8.4e-8.  (8^3 and 16^3 FP64 J x and residual: 3 %
//   less time.)
template <class S>
struct Dif {
    S o, p, q;
    __device__ __forceinline__ Dif(S u, const Line<S>& l) : o(u), p(sub2(shfl(u, l.n1), u)), q(sub2(shfl(u, l.n2), u)) {}
    __device__ __forceinline__ S val(const Line<S>& l) const { return fma3(l.L[2], q, fma3(l.L[1], p, o)); }
    __device__ __forceinline__ S der(const Line<S>& l) const { return fma3(l.D[2], q, mul2(l.D[1], p)); }
    // u_0 - 2 u_1 + u_2, the second derivative at every point of the line
    __device__ __forceinline__ S sec(const Line<S>& l) const {
        return fma3(splat<S>(l.d == 1 ? 1.0 : -2.0), l.d == 0 ? p : q, l.d == 0 ? q : p);
    }
};
// transpose of sec, with the weights: node a collects (1, -2, 1)_a times the line's weighted sum
template <class S>
__device__ __forceinline__ S sec_t(S u, const Line<S>& l) {
    const S w[3] = {splat<S>(gw(l.d)), splat<S>(gw((l.d + 1) % 3)), splat<S>(gw((l.d + 2) % 3))};
    const S s = fma3(w[2], shfl(u, l.n2), fma3(w[1], shfl(u, l.n1), mul2(w[0], u)));
    return l.d == 1 ? mul2(splat<S>(-2.0), s) : s;
}

// value, D_k gradient; HS: mixed (h) and pure (hd) second derivatives; LP: Laplacian
template <int D, bool HS, bool LP, class S>
__device__ __forceinline__ void q2_vgrad(S u, const Line<S> l[D], S& val, S g[D], S* h, S* hd, S* lap) {
    using Along = std::conditional_t<HS, Dif<S>, Tri<S>>;   // Tri: the value alone
    const Dif<S> t(u, l[0]);
    const S A = t.val(l[0]), B = t.der(l[0]);
    const Dif<S> ta(A, l[1]);
    const Along tb(B, l[1]);
    const S AA = ta.val(l[1]), AB = ta.der(l[1]), BA = tb.val(l[1]);
    S EA, AE;
    if (HS || LP) {
        EA = Tri<S>(t.sec(l[0]), l[1]).val(l[1]);
        AE = ta.sec(l[1]);
    }
    if constexpr (D == 2) {
        val = AA;
        g[0] = BA;
        g[1] = AB;
        if (HS) {
            h[0] = tb.der(l[1]);
            hd[0] = EA;
            hd[1] = AE;
        }
        if (LP) *lap = add2(EA, AE);
    } else {
        const Dif<S> taa(AA, l[2]);
        const Along tab(AB, l[2]), tba(BA, l[2]);
        val = taa.val(l[2]);
        g[2] = taa.der(l[2]);
        g[1] = tab.val(l[2]);
        g[0] = tba.val(l[2]);
        if (HS) {
            h[0] = Tri<S>(tb.der(l[1]), l[2]).val(l[2]);
            h[1] = tba.der(l[2]);
            h[2] = tab.der(l[2]);
            hd[0] = Tri<S>(EA, l[2]).val(l[2]);
            hd[1] = Tri<S>(AE, l[2]).val(l[2]);
            hd[2] = taa.sec(l[2]);
        }
        if (LP) *lap = Tri<S>(add2(EA, AE), l[2]).val(l[2], taa.sec(l[2]));
    }
}
// transposes, l: transposed lines
template <int D, bool HS, bool LP, class S>
__device__ __forceinline__ S q2_vgradT(S val, const S g[D], const S* h, const S* hd, S lap, const Line<S> l[D]) {
    S AA, AB, BA, EA = splat<S>(0.0), AE = splat<S>(0.0), BB = splat<S>(0.0);
    if constexpr (D == 3) {
        AA = Tri<S>(g[2], l[2]).der(l[2], Tri<S>(val, l[2]).val(l[2]));
        AB = Tri<S>(g[1], l[2]).val(l[2]);
        BA = Tri<S>(g[0], l[2]).val(l[2]);
        if (HS) {
            AB = Tri<S>(h[2], l[2]).der(l[2], AB);
            BA = Tri<S>(h[1], l[2]).der(l[2], BA);
            BB = Tri<S>(h[0], l[2]).val(l[2]);
            EA = Tri<S>(hd[0], l[2]).val(l[2]);
            AE = Tri<S>(hd[1], l[2]).val(l[2]);
            AA = add2(AA, sec_t(hd[2], l[2]));
        }
        if (LP) {
            EA = AE = Tri<S>(lap, l[2]).val(l[2]);
            AA = add2(AA, sec_t(lap, l[2]));
        }
    } else {
        AA = val;
        AB = g[1];
        BA = g[0];
        if (HS) {
            BB = h[0];
            EA = hd[0];
            AE = hd[1];
        }
        if (LP) EA = AE = lap;
    }
    S A = Tri<S>(AB, l[1]).der(l[1], Tri<S>(AA, l[1]).val(l[1])), B = Tri<S>(BA, l[1]).val(l[1]);
    S r;
    if (HS) B = Tri<S>(BB, l[1]).der(l[1], B);
    if (HS || LP) {
        A = add2(A, sec_t(AE, l[1]));
        r = sec_t(Tri<S>(EA, l[1]).val(l[1]), l[0]);
        r = Tri<S>(A, l[0]).val(l[0], r);
    } else {
        r = Tri<S>(A, l[0]).val(l[0]);
    }
    return Tri<S>(B, l[0]).der(l[0], r);
}
template <int D, class S>
__device__ __forceinline__ S q2_value(S u, const Line<S> l[D]) {
#pragma unroll
    for (int k = 0; k < D; ++k) u = Tri<S>(u, l[k]).val(l[k]);
    return u;
}
// value and derivative along axis K, and the transpose
template <int D, int K, class S>
__device__ __forceinline__ void q2_vder(S u, const Line<S> l[D], S& val, S& g) {
    val = u;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        if (k > K) g = Tri<S>(g, l[k]).val(l[k]);
        if (k == K) {
            const Dif<S> t(val, l[k]);
            g = t.der(l[k]);
            val = t.val(l[k]);
        } else {
            val = Tri<S>(val, l[k]).val(l[k]);
        }
    }
}
template <int D, int K, class S>
__device__ __forceinline__ S q2_vderT(S val, S g, const Line<S> l[D]) {
#pragma unroll
    for (int k = D - 1; k >= 0; --k) {
        if (k == K) {
            val = Tri<S>(g, l[k]).der(l[k], Tri<S>(val, l[k]).val(l[k]));
        } else {
            val = Tri<S>(val, l[k]).val(l[k]);
            if (k > K) g = Tri<S>(g, l[k]).val(l[k]);
        }
    }
    return val;
}

template <class S>
struct Q2Params {
    PwConst<S> c;
    PwLevel<S> L;
    S inv_dt;
};
template <int D, class S>
Q2Params<S> q2_params(const PhysConst& pc, double h) {
    Q2Params<S> p;
    const double c6 = 1.0 / (pc.Pe * pc.Cn), s = 2.0 / h, kap = s * s, g = kap;
    p.c.alpha = splat<S>(pc.alpha);
    p.c.beta = splat<S>(pc.beta);
    p.c.c2 = splat<S>(pc.gamma * pc.inv_Re);
    p.c.c5 = splat<S>(pc.xi * pc.inv_Re);
    p.c.inv_Fr = splat<S>(pc.inv_Fr);
    p.c.td = splat<S>(2.0 * pc.inv_dt);
    p.c.c0 = splat<S>(pc.four_over_dt2);
    p.c.inv_We = splat<S>(pc.inv_We);
    p.c.gk = splat<S>(1.0);
    p.L.s = splat<S>(s);
    p.L.kap = splat<S>(kap);
    p.L.vol = splat<S>(D == 2 ? 0.25 * h * h : 0.125 * h * h * h);
    p.L.nak = splat<S>(-pc.alpha * kap * c6);
    p.L.km = splat<S>(kap * c6);
    p.L.nc2k = splat<S>(-pc.gamma * pc.inv_Re * kap);
    p.L.cnk = splat<S>(pc.Cn * kap);
    p.L.cn2k = splat<S>(pc.Cn * pc.Cn * kap);
    p.L.c3 = splat<S>(pc.C_I * D * g * g);
    p.L.c3x2 = splat<S>(2.0 * pc.C_I * D * g * g);
    p.L.c4 = splat<S>(pc.C_phi * D * g * g * c6 * c6);
    p.L.c0p = splat<S>(pc.four_over_dt2 + pc.C_phi * D * g * g * c6 * c6);
    p.L.ct = splat<S>(pc.inv_We / (D * g));
    p.inv_dt = splat<S>(pc.inv_dt);
    return p;
}

// averages and their derivatives at the lane's point (or, from half a tangent, their tangents)
template <int D, class S>
__device__ __forceinline__ void q2_averages(const S u[D + 3], S ps, const Line<S> l[D], S inv_We, PwIn<D, S>& X, S& p, S& mu) {
#pragma unroll
    for (int i = 0; i < D; ++i) q2_vgrad<D, false, true>(u[i], l, X.v[i], X.gv[i], (S*)nullptr, (S*)nullptr, &X.lapv[i]);
    q2_vgrad<D, false, false>(u[D], l, p, X.gp, (S*)nullptr, (S*)nullptr, (S*)nullptr);
    p = mul2(inv_We, p);
    q2_vgrad<D, true, false>(u[D + 1], l, X.phi, X.gq, X.H, X.Hd, (S*)nullptr);
    q2_vgrad<D, false, true>(u[D + 2], l, mu, X.gm, (S*)nullptr, (S*)nullptr, &X.lapmu);
    q2_vgrad<D, false, false>(ps, l, X.ps, X.gs, (S*)nullptr, (S*)nullptr, (S*)nullptr);
}

// element of a warp's slot and half, and the lane's place in it
template <int D, class S>
struct Place {
    int idx;              // node / Gauss point
    bool active;
    int64_t e[Halves<S>::n];
    bool valid[Halves<S>::n];
    __device__ __forceinline__ Place(int64_t E) {
        constexpr int H = Halves<S>::n;
        const int lane = threadIdx.x & 31;
        const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        active = lane < 27;
        idx = active ? lane % Q2S<D>::NN : 0;
        const int64_t first = (warp * Q2S<D>::EPW + (active ? lane / Q2S<D>::NN : 0)) * H;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            valid[h] = active && first + h < E;
            e[h] = first + h < E ? first + h : E - 1;   // repeats the last element, adds nothing
        }
    }
};

enum { Q2_RES = 0, Q2_JVP = 1 };

template <int D, class S, int MODE>
__global__ void __launch_bounds__(Q2_THREADS, sizeof(typename Scalar<S>::type) == 4 ? 3 : 2)
q2_rj_kernel(DevMesh m, const __grid_constant__ Q2Params<S> prm, const typename Scalar<S>::type* __restrict__ Uo,
             const typename Scalar<S>::type* __restrict__ Un, const typename Scalar<S>::type* __restrict__ xin,
             typename Scalar<S>::type* __restrict__ out, unsigned int* __restrict__ flags, int pair_rows) {
    using T = typename Scalar<S>::type;
    constexpr int NN = Q2S<D>::NN, NF = Q2S<D>::NF, H = Halves<S>::n;
    const Place<D, S> P(m.E);
    const int lane = threadIdx.x & 31;
    int node[H];
    S u[NF], dd[D + 1], ps, x[NF], xps;
    {
        T gu[NF][H], gd[D + 1][H], gs[H], gx[NF][H], gxp[H];
#pragma unroll
        for (int h = 0; h < H; ++h) node[h] = __ldg(m.e2n + P.e[h] * NN + P.idx);
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const size_t r = (size_t)node[h] * NF;
            T o[NF], n[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                o[f] = __ldg(Uo + r + f);
                n[f] = __ldg(Un + r + f);
                if (MODE == Q2_JVP) gx[f][h] = T(0.5) * __ldg(xin + r + f);
            }
#pragma unroll
            for (int f = 0; f < NF; ++f) gu[f][h] = T(0.5) * (o[f] + n[f]);
#pragma unroll
            for (int i = 0; i < D; ++i) gd[i][h] = n[i] - o[i];
            gd[D][h] = n[D + 1] - o[D + 1];
            const T avg = gu[D + 1][h];
            const bool hi = avg > T(1), lo = avg < T(-1);
            gs[h] = hi ? T(1) : (lo ? T(-1) : avg);
            if (MODE == Q2_JVP) gxp[h] = hi || lo ? T(0) : gx[D + 1][h];
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            u[f] = pack(gu[f]);
            if (MODE == Q2_JVP) x[f] = pack(gx[f]);
        }
#pragma unroll
        for (int i = 0; i <= D; ++i) dd[i] = pack(gd[i]);
        ps = pack(gs);
        if (MODE == Q2_JVP) xps = pack(gxp);
    }
    const PwLevel<S>& L = prm.L;
    S sg[D];
#pragma unroll
    for (int k = 0; k < D; ++k) sg[k] = L.s;
    S F0[NF], F1[NF][D];
    {
        Line<S> l[D];
        int stride = 1;
#pragma unroll
        for (int k = 0; k < D; ++k, stride *= 3) l[k] = line<false, S>(lane, P.idx, stride, P.active);
        PwState<D, S> st;
        PwIn<D, S> X;
        S p, mu, ddiv = splat<S>(0.0);
        q2_averages<D, S>(u, ps, l, prm.c.inv_We, X, p, mu);
        if (MODE == Q2_RES) {
            S g;
            q2_vder<D, 0>(dd[0], l, X.a[0], g);
            ddiv = g;
            q2_vder<D, 1>(dd[1], l, X.a[1], g);
            ddiv = add2(ddiv, g);
            if constexpr (D == 3) {
                q2_vder<D, 2>(dd[2], l, X.a[2], g);
                ddiv = add2(ddiv, g);
            }
            ddiv = mul2(mul2(splat<S>(0.5), L.s), ddiv);
        } else {
#pragma unroll
            for (int i = 0; i < D; ++i) X.a[i] = q2_value<D>(dd[i], l);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) X.a[i] = mul2(prm.inv_dt, X.a[i]);
        X.pdt = mul2(prm.inv_dt, q2_value<D>(dd[D], l));
        const S pdt = X.pdt;
        pw_primal<D, S, true>(X, prm.c, L, sg, st);
        if constexpr (MODE == Q2_RES) {
            if (P.valid[0] && is_nan(st.Sh[0])) atomicOr(flags, 1u);
            pw_flux<D, S>(st, p, mu, pdt, add2(st.Rc, ddiv), prm.c, L, sg, F0, F1);
        } else {
            PwIn<D, S> dX;
            S dp, dmu;
            q2_averages<D, S>(x, xps, l, prm.c.inv_We, dX, dp, dmu);
            pw_tangent<D, S, true>(st, dX, dp, dmu, prm.c, L, sg, F0, F1);
        }
    }
    S r[NF];
    {
        Line<S> l[D];
        int stride = 1;
#pragma unroll
        for (int k = 0; k < D; ++k, stride *= 3) l[k] = line<true, S>(lane, P.idx, stride, P.active);
#pragma unroll
        for (int f = 0; f < NF; ++f)
            r[f] = mul2(L.vol, q2_vgradT<D, false, false, S>(F0[f], F1[f], nullptr, nullptr, splat<S>(0.0), l));
    }
    chain_wait<true>();
#pragma unroll
    for (int h = 0; h < H; ++h) {
        if (!P.valid[h]) continue;
        const unsigned skip = replaced_rows<D>(m, node[h], 0);
        T* o = out + (size_t)node[h] * NF;
        if constexpr (D == 3 && sizeof(T) == 4) {
            if (pair_rows && skip == 0) {
#pragma unroll
                for (int f = 0; f < NF; f += 2)
                    atomicAdd(reinterpret_cast<float2*>(o + f), make_float2(half_of(r[f], h), half_of(r[f + 1], h)));
                continue;
            }
        }
#pragma unroll
        for (int f = 0; f < NF; ++f)
            if (f >= D || !((skip >> f) & 1u)) atomicAdd(o + f, half_of(r[f], h));
    }
}

// J^T w on Q2 (FP64): seeds at the Gauss points, the adjoint of the pointwise map, the transpose of
// the interpolation
template <int D>
__global__ void __launch_bounds__(Q2_THREADS, 2)
q2_vjp_kernel(DevMesh m, const __grid_constant__ Q2Params<double> prm, double iCn, const double* __restrict__ Uo,
              const double* __restrict__ Un, const double* __restrict__ w, double* __restrict__ gn, double* __restrict__ go,
              double* __restrict__ gCn) {
    using S = double;
    constexpr int NN = Q2S<D>::NN, NF = Q2S<D>::NF;
    const Place<D, S> P(m.E);
    const int lane = threadIdx.x & 31;
    const int node = __ldg(m.e2n + P.e[0] * NN + P.idx);
    const PwLevel<S>& L = prm.L;
    S sg[D];
#pragma unroll
    for (int k = 0; k < D; ++k) sg[k] = L.s;
    bool inside;
    double cnb;
    PwIn<D, S> B;
    S pb, mub, divb;
    {
        Line<S> l[D];
        int stride = 1;
#pragma unroll
        for (int k = 0; k < D; ++k, stride *= 3) l[k] = line<false, S>(lane, P.idx, stride, P.active);
        PwState<D, S> st;
        {
            S u[NF], dd[D + 1], ps, p, mu;
            const size_t r = (size_t)node * NF;
            {
                S o[NF], n[NF];
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    o[f] = __ldg(Uo + r + f);
                    n[f] = __ldg(Un + r + f);
                    u[f] = 0.5 * (o[f] + n[f]);
                }
#pragma unroll
                for (int i = 0; i < D; ++i) dd[i] = n[i] - o[i];
                dd[D] = n[D + 1] - o[D + 1];
            }
            const bool hi = u[D + 1] > 1.0, lo = u[D + 1] < -1.0;
            inside = !(hi || lo);
            ps = hi ? 1.0 : (lo ? -1.0 : u[D + 1]);
            PwIn<D, S> X;
            q2_averages<D, S>(u, ps, l, prm.c.inv_We, X, p, mu);
#pragma unroll
            for (int i = 0; i < D; ++i) X.a[i] = prm.inv_dt * q2_value<D>(dd[i], l);
            X.pdt = prm.inv_dt * q2_value<D>(dd[D], l);
            pw_primal<D, S, true>(X, prm.c, L, sg, st);
        }
        S F0[NF], F1[NF][D];
        // seeds: Dirichlet rows are replaced rows, their element contributions are discarded
        const unsigned fl = replaced_rows<D>(m, node, 0);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            S wv = __ldg(w + (size_t)node * NF + f);
            if (f < D && ((fl >> f) & 1u)) wv = 0.0;
            q2_vgrad<D, false, false>(wv, l, F0[f], F1[f], (S*)nullptr, (S*)nullptr, (S*)nullptr);
        }
        pw_adjoint<D, S, true>(st, F0, F1, prm.c, L, sg, iCn, B, pb, mub, divb, cnb);
    }
    S rn[NF], ro[NF], psb, dt[D + 1];
    {
        Line<S> l[D];
        int stride = 1;
#pragma unroll
        for (int k = 0; k < D; ++k, stride *= 3) l[k] = line<true, S>(lane, P.idx, stride, P.active);
#pragma unroll
        for (int i = 0; i < D; ++i) {
            B.gv[i][i] = fma(L.s, divb, B.gv[i][i]);
            rn[i] = q2_vgradT<D, false, true, S>(B.v[i], B.gv[i], nullptr, nullptr, B.lapv[i], l);
        }
        rn[D] = q2_vgradT<D, false, false, S>(prm.c.inv_We * pb, B.gp, nullptr, nullptr, 0.0, l);
        rn[D + 1] = q2_vgradT<D, true, false, S>(B.phi, B.gq, B.H, B.Hd, 0.0, l);
        rn[D + 2] = q2_vgradT<D, false, true, S>(mub, B.gm, nullptr, nullptr, B.lapmu, l);
        psb = 0.5 * L.vol * q2_vgradT<D, false, false, S>(B.ps, B.gs, nullptr, nullptr, 0.0, l);
        // div v^{k+1} is div v~ plus half the difference's divergence
        const S hd = 0.5 * L.s * divb;
        dt[0] = q2_vderT<D, 0>(prm.inv_dt * B.a[0], hd, l);
        dt[1] = q2_vderT<D, 1>(prm.inv_dt * B.a[1], hd, l);
        if constexpr (D == 3) dt[2] = q2_vderT<D, 2>(prm.inv_dt * B.a[2], hd, l);
        S b = prm.inv_dt * B.pdt;
#pragma unroll
        for (int k = D - 1; k >= 0; --k) b = Tri<S>(b, l[k]).val(l[k]);
        dt[D] = b;
    }
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const S a = 0.5 * L.vol * rn[k];
        if (k == D || k == D + 2) {
            rn[k] = ro[k] = a;
        } else {
            const S b = dt[k < D ? k : D];
            rn[k] = fma(L.vol, b, a);
            ro[k] = fma(-L.vol, b, a);
        }
    }
    chain_wait<true>();
    if (P.valid[0]) {
        if (inside) {
            rn[D + 1] += psb;
            ro[D + 1] += psb;
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            atomicAdd(gn + (size_t)node * NF + f, rn[f]);
            if (go) atomicAdd(go + (size_t)node * NF + f, ro[f]);
        }
    }
    if (gCn) {
        int q = P.idx;
        S wq = L.vol;
#pragma unroll
        for (int k = 0; k < D; ++k, q /= 3) wq *= gw(q % 3);
        cnb = P.valid[0] ? cnb * wq : 0.0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) cnb += __shfl_xor_sync(0xffffffffu, cnb, off);
        if (lane == 0 && cnb != 0.0) atomicAdd(gCn, cnb);
    }
}

// blocks of four warps, or of one where those would leave SMs without a block
template <int D, int H>
void q2_grid(int64_t E, unsigned& blocks, int& threads) {
    const int64_t per = Q2S<D>::EPW * H, warps = (E + per - 1) / per;
    threads = warps < 16 * (int64_t)chns_num_sms() ? 32 : Q2_THREADS;
    blocks = (unsigned)((warps * 32 + threads - 1) / threads);
}

template <int D, class S, int MODE>
cudaError_t q2_launch_rj(const chns_mesh* mm, const PhysConst& pc, const typename Scalar<S>::type* Uo,
                         const typename Scalar<S>::type* Un, const typename Scalar<S>::type* x,
                         typename Scalar<S>::type* out, cudaStream_t s) {
    using T = typename Scalar<S>::type;
    const DevMesh& m = mm->dm;
    const cudaError_t err = launch_init_rows<D, T, MODE>(m, MODE == Q2_RES ? Un : x, Uo, out, nullptr, nullptr, 0, s);
    if (err != cudaSuccess) return err;
    unsigned blocks;
    int th;
    q2_grid<D, Halves<S>::n>(m.E, blocks, th);
    chain<true>(q2_rj_kernel<D, S, MODE>, blocks, th, s, m, q2_params<D, S>(pc, ldexp(m.hi - m.lo, -(int)mm->q2_level)), Uo, Un, x,
                                                   out, mm->d_flags, (uintptr_t)out % 8 == 0);
    chns_count_launches(1);
    return cudaGetLastError();
}
template <int D>
cudaError_t q2_launch_vjp_d(const chns_mesh* mm, const PhysConst& pc, const double* Uo, const double* Un, const double* w,
                            double* gn, double* go, double* gCn, cudaStream_t s) {
    const DevMesh& m = mm->dm;
    const cudaError_t err = launch_init_rows<D, double, ROWS_VJP>(m, w, nullptr, gn, go, gCn, 0, s);
    if (err != cudaSuccess) return err;
    unsigned blocks;
    int th;
    q2_grid<D, 1>(m.E, blocks, th);
    chain<true>(q2_vjp_kernel<D>, blocks, th, s, m, q2_params<D, double>(pc, ldexp(m.hi - m.lo, -(int)mm->q2_level)), 1.0 / pc.Cn, Uo,
                                           Un, w, gn, go, gCn);
    chns_count_launches(1);
    return cudaGetLastError();
}

}  // namespace

cudaError_t q2_launch_residual(const chns_mesh* m, const PhysConst& pc, const double* Uo, const double* Un, double* R,
                               cudaStream_t s) {
    return m->dm.dim == 2 ? q2_launch_rj<2, double, Q2_RES>(m, pc, Uo, Un, nullptr, R, s)
                          : q2_launch_rj<3, double, Q2_RES>(m, pc, Uo, Un, nullptr, R, s);
}
cudaError_t q2_launch_jvp64(const chns_mesh* m, const PhysConst& pc, const double* Uo, const double* Un,
                            const double* x, double* y, cudaStream_t s) {
    return m->dm.dim == 2 ? q2_launch_rj<2, double, Q2_JVP>(m, pc, Uo, Un, x, y, s)
                          : q2_launch_rj<3, double, Q2_JVP>(m, pc, Uo, Un, x, y, s);
}
cudaError_t q2_launch_jvp32(const chns_mesh* m, const PhysConst& pc, const float* Uo, const float* Un, const float* x,
                            float* y, cudaStream_t s) {
    return m->dm.dim == 2 ? q2_launch_rj<2, float2, Q2_JVP>(m, pc, Uo, Un, x, y, s)
                          : q2_launch_rj<3, float2, Q2_JVP>(m, pc, Uo, Un, x, y, s);
}
cudaError_t q2_launch_vjp(const chns_mesh* mm, const PhysConst& pc, const double* Uo, const double* Un,
                          const double* w, double* gn, double* go, double* gCn, cudaStream_t s) {
    return mm->dm.dim == 2 ? q2_launch_vjp_d<2>(mm, pc, Uo, Un, w, gn, go, gCn, s)
                           : q2_launch_vjp_d<3>(mm, pc, Uo, Un, w, gn, go, gCn, s);
}
