// Q1 element work shared by the residual, J x, J^T w and block-Jacobi kernels: gather of the
// element corners (with hanging-node constraints), sum-factorised interpolation to the Gauss
// points and its transpose, both by lane exchange.
//
// Lane mapping.  A lane owns Gauss point q and corner q of one element (S = double), or the
// two that differ in x (S = float2): 2^d or 2^(d-1) neighbouring lanes make an element.  The
// Q1 interpolation is applied one axis at a time between lanes that differ in that axis's
// bit: with the 1D weights c_+ (own corner) and c_- (the other), c_+ (u + r u') needs one
// fused multiply-add per value (r = c_-/c_+; the factor c_+^d is taken once, from the value) and
// u - u' is the derivative along the axis, up to its sign and scale.
// Value and gradient of a field take 9 operations per point in 3D; summing basis products,
// or each thread reducing all 8 corners by itself, takes 25 and more, which on the FP64 pipe
// (2 lanes per SM and clock) cost more than the whole exchange through the shuffle unit.
// The transpose runs the same exchanges backwards (12 operations, the value's scale included).
#pragma once

#include <cuda_runtime.h>

#include "chns_internal.h"
#include "point_physics.cuh"

constexpr double Q1_CP = 0.78867513459481288225;   // (1 + 1/sqrt 3)/2
constexpr double Q1_R = 0.26794919243112270647;    // (1 - 1/sqrt 3)/(1 + 1/sqrt 3) = 2 - sqrt 3
constexpr int Q1_LEVELS = 21;                      // element levels 0..20

template <int D>
struct Shape {
    static constexpr int NC = 1 << D;      // corners = Gauss points
    static constexpr int NF = D + 3;       // fields
    static constexpr int NH = (D == 2) ? 1 : 3;
};

// points per lane, lane-bit masks of the axes, type of an x derivative (equal at the two
// points of a float2 lane)
template <class S> struct Lanes;
template <> struct Lanes<double> {
    static constexpr int NP = 1, X = 1, Y = 2, Z = 4;
    using XD = double;
};
template <> struct Lanes<float2> {
    static constexpr int NP = 2, X = 0, Y = 1, Z = 2;
    using XD = float;
};

// 2^k, |k| < 1022
__device__ __forceinline__ double pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }

__device__ __forceinline__ double shx(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ float shx(float v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ float2 shx(float2 v, int m) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
// an x derivative at both points of a lane, and its transpose
__device__ __forceinline__ double xd_spread(double b) { return b; }
__device__ __forceinline__ float2 xd_spread(float b) { return make_float2(b, b); }
__device__ __forceinline__ double xd_fold(double b) { return b; }
__device__ __forceinline__ float xd_fold(float2 b) { return b.x + b.y; }

// u + r u' and u - u' along x
__device__ __forceinline__ void x_stage(double u, double& a, double& b) {
    const double o = shx(u, 1);
    a = fma(Q1_R, o, u);
    b = u - o;
}
__device__ __forceinline__ void x_stage(float2 u, float2& a, float& b) {
    a = fma3(splat<float2>(Q1_R), make_float2(u.y, u.x), u);
    b = u.y - u.x;
}
__device__ __forceinline__ double x_stageT(double a, double b) { return (a + b) + shx(fma(Q1_R, a, -b), 1); }
__device__ __forceinline__ float2 x_stageT(float2 a, float b) {
    const float2 t = fma3(splat<float2>(Q1_R), make_float2(a.y, a.x), a);
    return make_float2(t.x - b, t.y + b);
}
__device__ __forceinline__ double x_lerp(double u) { return fma(Q1_R, shx(u, 1), u); }
__device__ __forceinline__ float2 x_lerp(float2 u) { return fma3(splat<float2>(Q1_R), make_float2(u.y, u.x), u); }
// along y or z (lane mask m)
template <class V>
__device__ __forceinline__ V lerp(V u, int m) { return fma3(splat<V>(Q1_R), shx(u, m), u); }
template <class V>
__device__ __forceinline__ void stage(V u, int m, V& a, V& b) {
    const V o = shx(u, m);
    a = fma3(splat<V>(Q1_R), o, u);
    b = sub2(u, o);
}
template <class V>
__device__ __forceinline__ V stageT(V a, V b, int m) { return add2(add2(a, b), shx(fma3(splat<V>(Q1_R), a, neg1(b)), m)); }
// the same for a = f v: f and fr = f r
template <class V>
__device__ __forceinline__ V stageT(V f, V fr, V v, V b, int m) { return add2(fma3(f, v, b), shx(fma3(fr, v, neg1(b)), m)); }

// value, D_k gradient and (WH) mixed second derivatives at this lane's points
template <int D, bool WH, class S>
__device__ __forceinline__ void q1_vgrad(S u, S& val, S g[D], S* h) {
    using B = typename Lanes<S>::XD;
    constexpr int MY = Lanes<S>::Y, MZ = Lanes<S>::Z;
    S a, aa, ab;
    B b, ba, bb = B();
    x_stage(u, a, b);
    stage(a, MY, aa, ab);
    if (WH) stage(b, MY, ba, bb);
    else ba = lerp(b, MY);
    if constexpr (D == 2) {
        val = aa;
        g[0] = xd_spread(ba);
        g[1] = ab;
        if (WH) h[0] = xd_spread(bb);
    } else {
        stage(aa, MZ, val, g[2]);
        if (WH) {
            B t, tz;
            stage(ab, MZ, g[1], h[2]);
            stage(ba, MZ, t, tz);
            g[0] = xd_spread(t);
            h[1] = xd_spread(tz);
            h[0] = xd_spread(lerp(bb, MZ));
        } else {
            g[1] = lerp(ab, MZ);
            g[0] = xd_spread(lerp(ba, MZ));
        }
    }
}
template <int D, class S>
__device__ __forceinline__ S q1_value(S u) {
    S a = lerp(x_lerp(u), Lanes<S>::Y);
    if constexpr (D == 3) a = lerp(a, Lanes<S>::Z);
    return a;
}
// value and the derivative along axis K alone
template <int D, int K, class S>
__device__ __forceinline__ void q1_vder(S u, S& val, S& g) {
    constexpr int MY = Lanes<S>::Y, MZ = Lanes<S>::Z;
    if constexpr (K == 0) {
        typename Lanes<S>::XD b;
        S a;
        x_stage(u, a, b);
        a = lerp(a, MY);
        b = lerp(b, MY);
        if constexpr (D == 3) {
            a = lerp(a, MZ);
            b = lerp(b, MZ);
        }
        val = a;
        g = xd_spread(b);
    } else if constexpr (K == 1) {
        S a, b;
        stage(x_lerp(u), MY, a, b);
        if constexpr (D == 3) {
            a = lerp(a, MZ);
            b = lerp(b, MZ);
        }
        val = a;
        g = b;
    } else {
        stage(lerp(x_lerp(u), MY), MZ, val, g);
    }
}
// transposes: corner value from point cotangents (f val, g, h); fr = f r
template <int D, bool WH, class S>
__device__ __forceinline__ S q1_vgradT(S f, S fr, S val, const S g[D], const S* h) {
    using B = typename Lanes<S>::XD;
    constexpr int MY = Lanes<S>::Y, MZ = Lanes<S>::Z;
    S a, ab = g[1];
    B ba = xd_fold(g[0]), bb = B();
    if constexpr (D == 3) {
        const S aa = stageT(f, fr, val, g[2], MZ);
        if (WH) {
            ab = stageT(g[1], h[2], MZ);
            ba = stageT(ba, xd_fold(h[1]), MZ);
            bb = lerp(xd_fold(h[0]), MZ);
        } else {
            ab = lerp(ab, MZ);
            ba = lerp(ba, MZ);
        }
        a = stageT(aa, ab, MY);
    } else {
        if (WH) bb = xd_fold(h[0]);
        a = stageT(f, fr, val, ab, MY);
    }
    const B b = WH ? stageT(ba, bb, MY) : lerp(ba, MY);
    return x_stageT(a, b);
}
template <int D, int K, class S>
__device__ __forceinline__ S q1_vderT(S val, S g) {
    constexpr int MY = Lanes<S>::Y, MZ = Lanes<S>::Z;
    if constexpr (K == 0) {
        typename Lanes<S>::XD b = xd_fold(g);
        if constexpr (D == 3) {
            val = lerp(val, MZ);
            b = lerp(b, MZ);
        }
        return x_stageT(lerp(val, MY), lerp(b, MY));
    } else if constexpr (K == 1) {
        if constexpr (D == 3) {
            val = lerp(val, MZ);
            g = lerp(g, MZ);
        }
        return x_lerp(stageT(val, g, MY));
    } else {
        return x_lerp(lerp(stageT(val, g, MZ), MY));
    }
}

// ---- constants ------------------------------------------------------------------------
// Nodal data enter as sums of the two levels (and twice phi*), so a value is f = c_+^d/2 times
// the exchange's and a gradient s_j = +-f/(h c_+) times.
template <class S>
struct Q1Params {
    PwConst<S> c;
    S f, fr, inv_f;          // f, f r, 1/f
    S fc, fcr;               // f and f r of the test contraction, which rounds against f: f fc = f^2
    S sp;                    // f/We
    S sd;                    // scale of time differences: c_+^d/dt
    PwLevel<S> lev[Q1_LEVELS];
};
template <int D, class S>
Q1Params<S> q1_params(const PhysConst& pc, double span, int max_level) {
    Q1Params<S> p;
    const double cd = D == 2 ? Q1_CP * Q1_CP : Q1_CP * Q1_CP * Q1_CP, f = 0.5 * cd;
    const double c6 = 1.0 / (pc.Pe * pc.Cn);
    p.c.alpha = splat<S>(pc.alpha);
    p.c.beta = splat<S>(pc.beta);
    p.c.c2 = splat<S>(pc.gamma * pc.inv_Re);
    p.c.c5 = splat<S>(pc.xi * pc.inv_Re);
    p.c.inv_Fr = splat<S>(pc.inv_Fr);
    p.c.td = splat<S>(2.0 * pc.inv_dt);
    p.c.c0 = splat<S>(pc.four_over_dt2);
    p.c.inv_We = splat<S>(pc.inv_We);
    // s, s^2 and gk from powers of c_+, not from the rounded f: a constant's rounding is an error of every
    // entry alike (s^2 of f/c_+ in 2D: 2.1e-16), and so is that of f, which enters twice (2D FP32: -8.1e-8 with
    // f in both places, 1.5e-8 with fc)
    const double c = D == 2 ? Q1_CP : Q1_CP * Q1_CP;
    p.c.gk = splat<S>(16.0 / (c * c));
    const double fc = sizeof(typename Scalar<S>::type) == 4 ? f * f / (double)(float)f : f;
    p.f = splat<S>(f);
    p.fr = splat<S>(f * Q1_R);
    p.fc = splat<S>(fc);
    p.fcr = splat<S>(fc * Q1_R);
    p.inv_f = splat<S>(1.0 / f);
    p.sp = splat<S>(f * pc.inv_We);
    p.sd = splat<S>(cd * pc.inv_dt);
    for (int l = 0; l < Q1_LEVELS; ++l) {
        const double h = ldexp(span, -(l <= max_level ? l : max_level)), s = 0.5 * c / h, kap = 0.25 * (c * c) / (h * h);
        const double g = 4.0 / (h * h);
        PwLevel<S>& L = p.lev[l];
        L.s = splat<S>(s);
        L.kap = splat<S>(kap);
        L.vol = splat<S>(D == 2 ? 0.5 * h * h : 0.25 * h * h * h);   // |det J| c_+^d / f
        L.nak = splat<S>(-pc.alpha * kap * c6);
        L.km = splat<S>(kap * c6);
        L.nc2k = splat<S>(-pc.gamma * pc.inv_Re * kap);
        L.cnk = splat<S>(pc.Cn * kap);
        L.cn2k = splat<S>(pc.Cn * pc.Cn * kap);
        L.c3 = splat<S>(pc.C_I * D * g * g);
        L.c3x2 = splat<S>(2.0 * pc.C_I * D * g * g);
        L.c4 = splat<S>(pc.C_phi * D * g * g * c6 * c6);
        L.c0p = splat<S>(pc.four_over_dt2 + pc.C_phi * D * g * g * c6 * c6);
        L.ct = splat<S>(pc.inv_We / (D * g));
    }
    return p;
}

// the signed s_j of a lane's points (x: both signs are in a float2 lane's derivative itself)
template <int D, class S>
__device__ __forceinline__ void q1_signs(int lane_q, S s, S sg[D]) {
    using L = Lanes<S>;
    sg[0] = (L::NP == 2 || (lane_q & L::X)) ? s : neg1(s);
    sg[1] = (lane_q & L::Y) ? s : neg1(s);
    if constexpr (D == 3) sg[2] = (lane_q & L::Z) ? s : neg1(s);
}

// ---- gather ----------------------------------------------------------------------------
template <class T> struct Pair;
template <> struct Pair<float> { using type = float2; };
template <> struct Pair<double> { using type = double2; };

// A node row of NF values from global memory (read-only path).  In 3D a row is 24 B
// (FP32) or 48 B (FP64) at node * row, so it is read as three 8- or 16-byte pairs.
template <int D, class T>
__device__ __forceinline__ void ld_row(const T* __restrict__ p, T v[Shape<D>::NF]) {
    if constexpr (D == 3) {
        const typename Pair<T>::type* q = reinterpret_cast<const typename Pair<T>::type*>(p);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const typename Pair<T>::type t = __ldg(q + i);
            v[2 * i] = t.x;
            v[2 * i + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int f = 0; f < Shape<D>::NF; ++f) v[f] = __ldg(p + f);
    }
}

// Parents of an element corner: itself, or the 2 / 4 constraint parents of a hanging point.
struct Parents {
    int n;
    int4 p;
};
__device__ __forceinline__ Parents parents_of(const DevMesh& m, int ent) {
    Parents P;
    P.n = 1;
    P.p = make_int4(ent, 0, 0, 0);
    if (ent < 0) {
        P.p = __ldg(reinterpret_cast<const int4*>(m.hang) - ent - 1);
        P.n = P.p.z < 0 ? 2 : 4;
    }
    return P;
}
// j: a constant after unrolling
__device__ __forceinline__ int parent(const Parents& P, int j) { return j == 0 ? P.p.x : (j == 1 ? P.p.y : (j == 2 ? P.p.z : P.p.w)); }
template <class T>
__device__ __forceinline__ T parent_weight(int n) { return n == 1 ? T(1) : (n == 2 ? T(0.5) : T(0.25)); }

// phi* of a nodal average: the clip to [-1, 1]; inside: whether |phi~| <= 1 (NaN passes through)
template <class T>
__device__ __forceinline__ T clip_phi(T avg, bool& inside) {
    const bool hi = avg > T(1), lo = avg < T(-1);
    inside = !(hi || lo);
    return hi ? T(1) : (lo ? T(-1) : avg);
}

// The lane's NP corners: s = U^k + U^{k+1}, d = U^{k+1} - U^k of v and phi, ps = phi* (clipped at
// the independent nodes, then interpolated), twice, and, with TAN, the tangent row x and the
// tangent xps of twice phi* (x_phi where |phi~| <= 1).  The rows of every corner's first parent are loaded
// together, before anything depends on them: the gather's latency (not its bandwidth) is what
// the FP32 kernel waits for.  inside[h] bit j: parent j of corner h has |phi~| <= 1.
template <int D, int NP, bool TAN, class T>
__device__ __forceinline__ void gather_corners(const Parents P[NP], const T* __restrict__ Uo, const T* __restrict__ Un,
                                               const T* __restrict__ xin, T s[Shape<D>::NF][NP], T d[D + 1][NP],
                                               T ps[NP], T x[Shape<D>::NF][NP], T xps[NP], unsigned inside[NP]) {
    constexpr int NF = Shape<D>::NF;
    T o[NP][NF], n[NP][NF], xr[NP][NF];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        ld_row<D, T>(Uo + (size_t)P[h].p.x * NF, o[h]);
        ld_row<D, T>(Un + (size_t)P[h].p.x * NF, n[h]);
        if (TAN) ld_row<D, T>(xin + (size_t)P[h].p.x * NF, xr[h]);
    }
    bool more = false;
#pragma unroll
    for (int h = 0; h < NP; ++h) {
#pragma unroll
        for (int f = 0; f < NF; ++f) s[f][h] = o[h][f] + n[h][f];
#pragma unroll
        for (int i = 0; i < D; ++i) d[i][h] = n[h][i] - o[h][i];
        d[D][h] = n[h][D + 1] - o[h][D + 1];
        bool in;
        ps[h] = T(2) * clip_phi(T(0.5) * s[D + 1][h], in);
        inside[h] = in ? 1u : 0u;
        if (TAN) {
#pragma unroll
            for (int f = 0; f < NF; ++f) x[f][h] = xr[h][f];
            xps[h] = in ? xr[h][D + 1] : T(0);
        }
        more = more || P[h].n > 1;
    }
    if (more) {
#pragma unroll
        for (int h = 0; h < NP; ++h) {
#pragma unroll
            for (int j = 1; j < 4; ++j) {
                if (j >= P[h].n) continue;
                const size_t row = (size_t)parent(P[h], j) * NF;
                ld_row<D, T>(Uo + row, o[h]);
                ld_row<D, T>(Un + row, n[h]);
                if (TAN) ld_row<D, T>(xin + row, xr[h]);
#pragma unroll
                for (int f = 0; f < NF; ++f) s[f][h] += o[h][f] + n[h][f];
#pragma unroll
                for (int i = 0; i < D; ++i) d[i][h] += n[h][i] - o[h][i];
                d[D][h] += n[h][D + 1] - o[h][D + 1];
                bool in;
                ps[h] += T(2) * clip_phi(T(0.5) * (o[h][D + 1] + n[h][D + 1]), in);
                if (in) inside[h] |= 1u << j;
                if (TAN) {
#pragma unroll
                    for (int f = 0; f < NF; ++f) x[f][h] += xr[h][f];
                    if (in) xps[h] += xr[h][D + 1];
                }
            }
            const T w = parent_weight<T>(P[h].n);
#pragma unroll
            for (int f = 0; f < NF; ++f) s[f][h] *= w;
#pragma unroll
            for (int i = 0; i <= D; ++i) d[i][h] *= w;
            ps[h] *= w;
            if (TAN) {
#pragma unroll
                for (int f = 0; f < NF; ++f) x[f][h] *= w;
                xps[h] *= w;
            }
        }
    }
}
// the lane's corners as working values
__device__ __forceinline__ double pack(const double* a) { return a[0]; }
__device__ __forceinline__ float2 pack(const float* a) { return make_float2(a[0], a[1]); }
__device__ __forceinline__ float half_of(float2 v, int i) { return i == 0 ? v.x : v.y; }
__device__ __forceinline__ double half_of(double v, int) { return v; }

// Averages at the lane's points from the corners' sums s and twice phi* (ps): the inputs of the
// pointwise map, or (from x and its phi* tangent) their tangents.  PM: also the values of p/We
// and mu.
template <int D, bool PM, class S>
__device__ __forceinline__ void q1_averages(const Q1Params<S>& prm, const S s[D + 3], S ps, PwIn<D, S>& X, S& p, S& mu) {
    S t;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        q1_vgrad<D, false>(s[i], t, X.gv[i], (S*)nullptr);
        X.v[i] = mul2(prm.f, t);
    }
    q1_vgrad<D, false>(s[D], t, X.gp, (S*)nullptr);
    if (PM) p = mul2(prm.sp, t);
    q1_vgrad<D, true>(s[D + 1], t, X.gq, X.H);
    X.phi = mul2(prm.f, t);
#pragma unroll
    for (int k = 0; k < Shape<D>::NH; ++k) X.H[k] = mul2(prm.inv_f, X.H[k]);
    q1_vgrad<D, false>(s[D + 2], t, X.gm, (S*)nullptr);
    if (PM) mu = mul2(prm.f, t);
    q1_vgrad<D, false>(ps, t, X.gs, (S*)nullptr);
    X.ps = mul2(prm.f, t);
}
// Time differences at the lane's points from the corners' differences d.  DIV: also half the
// divergence of v^{k+1} - v^k (the solenoidality row acts on the new level).
template <int D, bool DIV, class S>
__device__ __forceinline__ void q1_differences(const Q1Params<S>& prm, const S sg[D], const S d[D + 1], PwIn<D, S>& X,
                                               S& ddiv) {
    if constexpr (DIV) {
        S t, g;
        q1_vder<D, 0>(d[0], t, g);
        X.a[0] = mul2(prm.sd, t);
        ddiv = mul2(sg[0], g);
        q1_vder<D, 1>(d[1], t, g);
        X.a[1] = mul2(prm.sd, t);
        ddiv = fma3(sg[1], g, ddiv);
        if constexpr (D == 3) {
            q1_vder<D, 2>(d[2], t, g);
            X.a[2] = mul2(prm.sd, t);
            ddiv = fma3(sg[2], g, ddiv);
        }
    } else {
#pragma unroll
        for (int i = 0; i < D; ++i) X.a[i] = mul2(prm.sd, q1_value<D>(d[i]));
    }
    X.pdt = mul2(prm.sd, q1_value<D>(d[D]));
}
