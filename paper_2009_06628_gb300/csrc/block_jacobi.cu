// Diagonal n_f x n_f block of J at every independent node: the sum over its element corners of
// d r_e[a] / d u_e[a], from the tangents of the corner's own basis function in every field.
// Hanging corners are skipped: the preconditioner is approximate there (it only affects
// convergence).  Also the element coefficients of the pressure Schur approximation.
//
// The lanes are those of the element kernels (one Gauss point per lane in FP64, two in FP32).
// Per corner and field the tangent of a basis function of one field alone (pw_unit) moves few
// of the pointwise terms; its test contraction with the same corner's basis is one number per
// row, and the n_f^2 numbers of a corner are summed over the element's lanes by recursive
// halving, which leaves each lane its own share of the block to add.
// 64^3: FP32 0.44 ms; 32^3: FP64 set-up in whole 3.1 ms (full dual-number map per field and
// corner, every number reduced to one lane before: 2.46 and about 12 ms).  Bound by the FP32 issue and
// the FP64 pipe.
#include <cuda_runtime.h>

#include "block_jacobi.h"
#include "point_physics.cuh"
#include "q1_lanes.cuh"

namespace {

__device__ __forceinline__ float fold(float2 v) { return v.x + v.y; }
__device__ __forceinline__ double fold(double v) { return v; }

// basis function of corner a at this lane's points, as the exchange of q1_lanes.cuh would leave it
// for unit data: value and D_k derivatives
template <int D>
__device__ __forceinline__ void unit_basis(int lane, int a, double& v, double g[D]) {
    double w[D], s[D];
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const bool own = ((a >> k) & 1) == ((lane >> k) & 1);
        w[k] = own ? 1.0 : Q1_R;
        s[k] = own ? 1.0 : -1.0;
    }
    v = D == 2 ? w[0] * w[1] : w[0] * w[1] * w[D - 1];
#pragma unroll
    for (int k = 0; k < D; ++k) {
        double p = s[k];
#pragma unroll
        for (int j = 0; j < D; ++j)
            if (j != k) p *= w[j];
        g[k] = p;
    }
}
template <int D>
__device__ __forceinline__ void unit_basis(int lane, int a, float2& v, float2 g[D]) {
    const float r = (float)Q1_R;
    const float wy = ((a >> 1) & 1) == (lane & 1) ? 1.0f : r, sy = ((a >> 1) & 1) == (lane & 1) ? 1.0f : -1.0f;
    const float wz = D == 2 ? 1.0f : ((a >> 2) == ((lane >> 1) & 1) ? 1.0f : r);
    const float2 wx = (a & 1) ? make_float2(r, 1.0f) : make_float2(1.0f, r);
    const float sx = (a & 1) ? 1.0f : -1.0f;
    v = make_float2(wx.x * wy * wz, wx.y * wy * wz);
    g[0] = make_float2(sx * wy * wz, sx * wy * wz);
    g[1] = make_float2(wx.x * sy * wz, wx.y * sy * wz);
    if constexpr (D == 3) {
        const float sz = (a >> 2) == ((lane >> 1) & 1) ? 1.0f : -1.0f;
        g[2] = make_float2(wx.x * wy * sz, wx.y * wy * sz);
    }
}
// mixed second derivatives of the same function (needed for phi)
template <int D>
__device__ __forceinline__ void unit_mixed(int lane, int a, double h[]) {
    double w[D], s[D];
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const bool own = ((a >> k) & 1) == ((lane >> k) & 1);
        w[k] = own ? 1.0 : Q1_R;
        s[k] = own ? 1.0 : -1.0;
    }
    h[0] = s[0] * s[1] * (D == 3 ? w[D - 1] : 1.0);
    if constexpr (D == 3) {
        h[1] = s[0] * w[1] * s[2];
        h[2] = w[0] * s[1] * s[2];
    }
}
template <int D>
__device__ __forceinline__ void unit_mixed(int lane, int a, float2 h[]) {
    const float r = (float)Q1_R;
    const bool oy = ((a >> 1) & 1) == (lane & 1);
    const float wy = oy ? 1.0f : r, sy = oy ? 1.0f : -1.0f;
    const bool oz = D == 2 || (a >> 2) == ((lane >> 1) & 1);
    const float wz = oz ? 1.0f : r, sz = oz ? 1.0f : -1.0f;
    const float2 wx = (a & 1) ? make_float2(r, 1.0f) : make_float2(1.0f, r);
    const float sx = (a & 1) ? 1.0f : -1.0f;
    h[0] = make_float2(sx * sy * (D == 3 ? wz : 1.0f), sx * sy * (D == 3 ? wz : 1.0f));
    if constexpr (D == 3) {
        h[1] = make_float2(sx * wy * sz, sx * wy * sz);
        h[2] = make_float2(wx.x * sy * sz, wx.y * sy * sz);
    }
}

// test contraction of one tangent with the corner's own basis: column F of the block
template <int D, int F, class S, class T>
__device__ __forceinline__ void column(const S F0[D + 3], const S F1[D + 3][D], S n, const S g[D], T* v) {
    constexpr int NF = D + 3;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        S r = mul2(n, F0[f]);
#pragma unroll
        for (int k = 0; k < D; ++k) r = fma3(g[k], F1[f][k], r);
        v[f * NF + F] = fold(r);
    }
}

template <int D, class S>
__global__ void __launch_bounds__(128, 2)
pc_build_kernel(DevMesh m, const __grid_constant__ Q1Params<S> prm, const typename Scalar<S>::type* __restrict__ Uo,
                const typename Scalar<S>::type* __restrict__ Un, typename Scalar<S>::type* __restrict__ blk,
                float* __restrict__ ce, double ce_scale) {
    using T = typename Scalar<S>::type;
    constexpr int NC = Shape<D>::NC, NF = Shape<D>::NF, NP = Lanes<S>::NP, LPE = NC / NP, NV = NF * NF;
    constexpr int NVP = (NV + LPE - 1) / LPE * LPE;   // padded to halve evenly
    const int t = threadIdx.x % LPE;
    const int64_t idx = (int64_t)blockIdx.x * (blockDim.x / LPE) + threadIdx.x / LPE;
    const bool valid = idx < m.E;
    const int64_t e = valid ? idx : m.E - 1;
    const PwLevel<S>& L = prm.lev[m.level[e]];
    int ent[NP];
    unsigned inside[NP];
    S sg[D];
    q1_signs<D>(t, L.s, sg);
    PwState<D, S> st;
    {
        T gs[NF][NP], gd[D + 1][NP], gp[NP], gx[NF][NP], gxp[NP];
        Parents P[NP];
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            ent[h] = m.e2n[e * NC + t * NP + h];
            P[h] = parents_of(m, ent[h]);
        }
        gather_corners<D, NP, false, T>(P, Uo, Un, nullptr, gs, gd, gp, gx, gxp, inside);
        S s[NF], d[D + 1], p, mu, dd;
        PwIn<D, S> X;
#pragma unroll
        for (int f = 0; f < NF; ++f) s[f] = pack(gs[f]);
#pragma unroll
        for (int i = 0; i <= D; ++i) d[i] = pack(gd[i]);
        q1_averages<D, false>(prm, s, pack(gp), X, p, mu);
        q1_differences<D, false>(prm, sg, d, X, dd);
        pw_primal<D, S, false>(X, prm.c, L, sg, st);
    }
    {
        // coefficient of the pressure Schur-complement approximation on this element:
        // dt/(2 We) times the mean of 1/rho(phi*) over the Gauss points
        T ir = fold(st.irho);
#pragma unroll
        for (int o = LPE / 2; o > 0; o >>= 1) ir += __shfl_xor_sync(0xffffffffu, ir, o);
        if (valid && t == 0) ce[e] = (float)(ce_scale * (double)ir / NC);
    }
    const T vol = half_of(L.vol, 0);
#pragma unroll 1
    for (int a = 0; a < NC; ++a) {
        T v[NVP];
#pragma unroll
        for (int i = NV; i < NVP; ++i) v[i] = T(0);
        S raw, n, g[D], F0[NF], F1[NF][D];
        unit_basis<D>(t, a, raw, g);
        n = mul2(prm.f, raw);
        pw_unit<D, S, 0>(st, n, g, prm.c, L, sg, F0, F1);
        column<D, 0>(F0, F1, n, g, v);
        pw_unit<D, S, 1>(st, n, g, prm.c, L, sg, F0, F1);
        column<D, 1>(F0, F1, n, g, v);
        if constexpr (D == 3) {
            pw_unit<D, S, 2>(st, n, g, prm.c, L, sg, F0, F1);
            column<D, 2>(F0, F1, n, g, v);
        }
        pw_unit<D, S, D>(st, n, g, prm.c, L, sg, F0, F1);
        column<D, D>(F0, F1, n, g, v);
        const int src = (threadIdx.x & 31 & ~(LPE - 1)) + a / NP;
        const unsigned in = __shfl_sync(0xffffffffu, NP == 2 && (a & 1) ? inside[NP - 1] : inside[0], src);
        {
            PwIn<D, S> X;
            const S z0 = splat<S>(0.0), on = splat<S>((in & 1u) ? 1.0 : 0.0);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                X.v[i] = X.gp[i] = X.gm[i] = z0;
#pragma unroll
                for (int k = 0; k < D; ++k) X.gv[i][k] = z0;
                X.gq[i] = g[i];
                X.gs[i] = mul2(on, g[i]);
            }
            X.phi = n;
            X.ps = mul2(on, n);
            unit_mixed<D>(t, a, X.H);
#pragma unroll
            for (int k = 0; k < Shape<D>::NH; ++k) X.H[k] = mul2(prm.inv_f, X.H[k]);
            pw_tangent<D, S, false>(st, X, z0, z0, prm.c, L, sg, F0, F1);
            column<D, D + 1>(F0, F1, n, g, v);
        }
        pw_unit<D, S, D + 2>(st, n, g, prm.c, L, sg, F0, F1);
        column<D, D + 2>(F0, F1, n, g, v);
        // sum over the element's lanes: each halving hands half of the numbers to the partner
        int base = 0, cnt = NVP;
#pragma unroll
        for (int o = LPE / 2; o > 0; o >>= 1) {
            cnt /= 2;
            const bool up = t & o;
#pragma unroll
            for (int i = 0; i < NVP / 2; ++i) {
                if (i >= cnt) break;
                const T keep = up ? v[cnt + i] : v[i], give = up ? v[i] : v[cnt + i];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
            base += up ? cnt : 0;
        }
        const int node = __shfl_sync(0xffffffffu, NP == 2 && (a & 1) ? ent[NP - 1] : ent[0], src);
        if (valid && node >= 0) {
            T* b = blk + (size_t)node * NV + base;
#pragma unroll
            for (int i = 0; i < NVP / LPE; ++i)
                if (base + i < NV) atomicAdd(b + i, vol * v[i]);
        }
    }
}

template <int D, class S>
cudaError_t launch(const chns_mesh* mm, const PhysConst& pc, const typename Scalar<S>::type* Uo,
                   const typename Scalar<S>::type* Un, typename Scalar<S>::type* blk, float* ce, cudaStream_t s) {
    using T = typename Scalar<S>::type;
    const DevMesh& m = mm->dm;
    cudaError_t e = cudaMemsetAsync(blk, 0, (size_t)m.N * m.nf * m.nf * sizeof(T), s);
    if (e != cudaSuccess) return e;
    const int64_t lanes = m.E * (Shape<D>::NC / Lanes<S>::NP);
    // one-warp blocks where four-warp ones would leave SMs idle (as the element kernels)
    const int th = lanes < (int64_t)512 * chns_num_sms() ? 32 : 128;
    pc_build_kernel<D, S><<<(unsigned)((lanes + th - 1) / th), th, 0, s>>>(
        m, q1_params<D, S>(pc, m.hi - m.lo, mm->max_level), Uo, Un, blk, ce, pc.dt / (2.0 * pc.We));
    chns_count_launches(1);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_pc_build(const chns_mesh* m, const PhysConst& pc, const float* Uo, const float* Un, float* blk,
                            float* ce, cudaStream_t s) {
    return m->dm.dim == 2 ? launch<2, float2>(m, pc, Uo, Un, blk, ce, s) : launch<3, float2>(m, pc, Uo, Un, blk, ce, s);
}
cudaError_t launch_pc_build(const chns_mesh* m, const PhysConst& pc, const double* Uo, const double* Un, double* blk,
                            float* ce, cudaStream_t s) {
    return m->dm.dim == 2 ? launch<2, double>(m, pc, Uo, Un, blk, ce, s) : launch<3, double>(m, pc, Uo, Un, blk, ce, s);
}
