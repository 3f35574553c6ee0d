// Element kernels of the matrix-free hot path: residual (FP64), J x (FP64 / FP32) and J^T w
// (FP64), each one pass over the elements: gather, interpolation, pointwise map (or its
// tangent / adjoint), test contraction, scatter.
//
// Lanes: 2^d per element in FP64 (lane q owns corner q and Gauss point q), 2^(d-1) in FP32
// (two corners / points per lane in packed arithmetic).  An element's lanes sit in one warp
// and exchange through shuffles only (q1_lanes.cuh); there is no shared memory and no barrier.
// Elements are processed in their Morton order (consecutive elements share most nodes, which
// keeps gathers in L2/L1).
//
// Hanging corners (Section 4): a corner value is the mean of its 2 (edge) or 4 (face)
// parent nodes; the scatter applies the transpose (the same weights).
//
// What bounds them: FP64, the FP64 pipe (2 lanes per SM and clock), so operations per Gauss
// point are the whole cost: lane-exchange interpolation and the regrouped pointwise map
// (point_physics.cuh) brought them, on 64^3 elements, from 925 / 1471 / 1753 to about 365 /
// 580 / 720 for the residual, J x and J^T w: 3.08 / 4.90 / 5.85 ms -> 1.39 / 2.25 / 2.60 ms
// (one thread per Gauss point with shared-memory corners and dual numbers before).
// FP32 J x: 543 instead of 1696 instructions per Gauss point (packed pairs); 64^3 135 -> 69 us,
// 128^3 997 -> 491 us per call.  It now waits for its gathers: 168 registers leave 12 warps per
// SM (ncu: half of the stall cycles on global loads, FMA pipe 40 %, shuffle/load unit 52 %).
// 2 or 4 resident blocks instead of 3: 128^3 571 / 716 us (484 at the time).
#include <cuda_runtime.h>

#include <type_traits>

#include "chns_internal.h"
#include "point_physics.cuh"
#include "q1_lanes.cuh"
#include "replaced_rows.cuh"

namespace {

constexpr int EK_THREADS = 128;

// Scatter strategies of the element kernels (chns_mesh_set_scatter):
//   SCAT_ATOMIC  one atomic add per corner row entry and parent (default);
//   SCAT_PLAIN   plain read-modify-write, for launches over one colour of an element
//                colouring (no two elements of a colour share a node): deterministic;
//   SCAT_WARPAGG the lanes of a warp that target the same node (found with
//                __match_any_sync) add their rows in shared memory first and one lane
//                issues the atomics.
enum { SCAT_ATOMIC = 0, SCAT_PLAIN = 1, SCAT_WARPAGG = 2 };

// Replaced rows (replaced_rows.cuh) were written before the launch and take no contribution.
// skip0: the replaced rows of the first parent (loaded with the gather).
// pair_rows: 3D FP32 rows (24 B) start on 8-byte boundaries of `out` and are added two entries
// per atomic.
template <int D, class T, int SCAT>
__device__ __forceinline__ void scatter_add(const DevMesh& m, T* __restrict__ out, const Parents& P,
                                            const T r[Shape<D>::NF], unsigned skip0, int pair_rows, int pin) {
    constexpr int NF = Shape<D>::NF;
    const T w = parent_weight<T>(P.n);
    if constexpr (SCAT == SCAT_PLAIN && sizeof(T) == 4) {
        // a corner's parents differ: all of their rows are on the way before the first is written (the FP64
        // kernels have no registers left for it)
        unsigned skip[4];
        T old[4][NF];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= P.n) break;
            skip[j] = j == 0 ? skip0 : replaced_rows<D>(m, parent(P, j), pin);
#pragma unroll
            for (int f = 0; f < NF; ++f) old[j][f] = out[(size_t)parent(P, j) * NF + f];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= P.n) break;
#pragma unroll
            for (int f = 0; f < NF; ++f)
                if (f > D || !((skip[j] >> f) & 1u)) out[(size_t)parent(P, j) * NF + f] = old[j][f] + w * r[f];
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (j >= P.n) break;
        const int node = parent(P, j);
        const unsigned skip = j == 0 ? skip0 : replaced_rows<D>(m, node, pin);
        T* o = out + (size_t)node * NF;
        if constexpr (D == 3 && sizeof(T) == 4 && SCAT == SCAT_ATOMIC) {
            if (pair_rows && skip == 0) {
#pragma unroll
                for (int f = 0; f < NF; f += 2)
                    atomicAdd(reinterpret_cast<float2*>(o + f), make_float2(w * r[f], w * r[f + 1]));
                continue;
            }
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            if (f <= D && ((skip >> f) & 1u)) continue;
            if (SCAT == SCAT_PLAIN)
                o[f] += w * r[f];
            else
                atomicAdd(o + f, w * r[f]);
        }
    }
}

// Plain adds of a warp's elements, LPE lanes each (SCAT_PLAIN; all lanes call it).  add(): this lane's rows;
// hanging: whether its corner is.  The corners of an element that are nodes are distinct, so they add
// together; a hanging corner's parents can be nodes of the element or another corner's parents, so
// those add one after another, in a fixed order.  FP32 J x, us, with all corners in turn / so / with the
// rows of scatter_add on the way together: 64^3 (8 colours) 320 / 263 / 173, a sphere on levels 3 to 6
// 750 / 685 / 515; one thread per corner took 295 and 543.
template <int LPE, class Add>
__device__ __forceinline__ void plain_adds(int t, bool valid, bool hanging, Add add) {
    if (valid && !hanging) add();
    __syncwarp();
    unsigned turns = __ballot_sync(0xffffffffu, valid && hanging);
#pragma unroll
    for (int o = LPE; o < 32; o <<= 1) turns |= turns >> o;
    for (turns &= (1u << LPE) - 1u; turns; turns &= turns - 1u) {
        if (valid && hanging && t == __ffs(turns) - 1) add();
        __syncwarp();
    }
}

// Warp-aggregated scatter: every lane of the warp calls it (valid == false: no rows).
// wbuf: this warp's 32 x NF shared staging rows.
template <int D, class T>
__device__ __forceinline__ void scatter_add_warpagg(const DevMesh& m, T* __restrict__ out, const Parents& P, const T r[Shape<D>::NF],
                                                    bool valid, T (*wbuf)[Shape<D>::NF], int pin) {
    constexpr int NF = Shape<D>::NF;
    const int lane = threadIdx.x & 31;
    const T w = parent_weight<T>(P.n);
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
        const int node = (valid && j < P.n) ? parent(P, j) : -1;
        if (node >= 0) {
#pragma unroll
            for (int f = 0; f < NF; ++f) wbuf[lane][f] = w * r[f];
        }
        __syncwarp();
        const unsigned grp = __match_any_sync(0xffffffffu, node);
        if (node >= 0 && lane == __ffs(grp) - 1) {
            T acc[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) acc[f] = T(0);
            for (unsigned g = grp; g; g &= g - 1) {
                const int src = __ffs(g) - 1;
#pragma unroll
                for (int f = 0; f < NF; ++f) acc[f] += wbuf[src][f];
            }
            T* o = out + (size_t)node * NF;
            const unsigned skip = replaced_rows<D>(m, node, pin);
#pragma unroll
            for (int f = 0; f < NF; ++f)
                if (f > D || !((skip >> f) & 1u)) atomicAdd(o + f, acc[f]);
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------------
// Residual (MODE_RES) and J x (MODE_JVP) share one kernel body.
// ---------------------------------------------------------------------------------
enum { MODE_RES = 0, MODE_JVP = 1 };

// resident blocks asked of the compiler
template <class S, int MODE>
constexpr int rj_blocks() { return sizeof(typename Scalar<S>::type) == 4 ? 3 : 2; }

template <int D, class S, int MODE, int SCAT>
__global__ void __launch_bounds__(EK_THREADS, (rj_blocks<S, MODE>()))
elem_rj_kernel(DevMesh m, const __grid_constant__ Q1Params<S> prm, const typename Scalar<S>::type* __restrict__ Uo,
               const typename Scalar<S>::type* __restrict__ Un, const typename Scalar<S>::type* __restrict__ xin,
               typename Scalar<S>::type* __restrict__ out, unsigned int* __restrict__ flags,
               const int32_t* __restrict__ elist, int64_t ecount, int pair_rows, int pin) {
    using T = typename Scalar<S>::type;
    constexpr int NC = Shape<D>::NC, NF = Shape<D>::NF, NP = Lanes<S>::NP, LPE = NC / NP;
    __shared__ T wbuf[SCAT == SCAT_WARPAGG ? EK_THREADS / 32 : 1][32][NF];
    const int t = threadIdx.x % LPE, le = threadIdx.x / LPE;
    const int64_t epb = blockDim.x / LPE, step = (int64_t)gridDim.x * epb;
    // element: the idx-th of the launch (elist: the listed elements of one colour); lanes past
    // the end repeat the last element and add nothing.  A block walks the launch with the
    // stride of the grid, the corner entries and level of its next elements loaded ahead.
    int ent_next[NP], lev_next;
    auto fetch = [&](int64_t i) {
        const int64_t ie = i < ecount ? i : ecount - 1;
        const int64_t e = elist ? (int64_t)elist[ie] : ie;
        lev_next = m.level[e];
#pragma unroll
        for (int h = 0; h < NP; ++h) ent_next[h] = __ldg(m.e2n + e * NC + t * NP + h);
    };
    int64_t idx = (int64_t)blockIdx.x * epb + le;
    fetch(idx);
    for (int64_t base = (int64_t)blockIdx.x * epb; base < ecount; base += step, idx += step) {
        const bool valid = idx < ecount;
        const PwLevel<S>& L = prm.lev[lev_next];
        int ent[NP];
#pragma unroll
        for (int h = 0; h < NP; ++h) ent[h] = ent_next[h];
        fetch(idx + step);
        S sg[D];
        q1_signs<D>(t, L.s, sg);

        S F0[NF], F1[NF][D];
        unsigned skips = 0;
        {
            PwState<D, S> st;
            PwIn<D, S> X;
            S p, mu, ddiv, xs[NF], xps;
            {
                T gs[NF][NP], gd[D + 1][NP], gp[NP], gx[NF][NP], gxp[NP];
                unsigned inside[NP];
                Parents P[NP];
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    P[h] = parents_of(m, ent[h]);
                    skips |= replaced_rows<D>(m, P[h].p.x, pin) << (8 * h);
                }
                gather_corners<D, NP, MODE == MODE_JVP, T>(P, Uo, Un, xin, gs, gd, gp, gx, gxp, inside);
                S s[NF], d[D + 1];
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    s[f] = pack(gs[f]);
                    if (MODE == MODE_JVP) xs[f] = pack(gx[f]);
                }
#pragma unroll
                for (int i = 0; i <= D; ++i) d[i] = pack(gd[i]);
                if (MODE == MODE_JVP) xps = pack(gxp);
                q1_averages<D, MODE == MODE_RES>(prm, s, pack(gp), X, p, mu);
                q1_differences<D, MODE == MODE_RES>(prm, sg, d, X, ddiv);
            }
            const S pdt = X.pdt;
            pw_primal<D, S, false>(X, prm.c, L, sg, st);
            if constexpr (MODE == MODE_RES) {
                // a non-positive tau_m radicand shows up as a non-finite tau
                if (valid && is_nan(st.Sh[0])) atomicOr(flags, 1u);
                S divnew = ddiv;
#pragma unroll
                for (int i = 0; i < D; ++i) divnew = fma3(sg[i], st.gv[i][i], divnew);
                pw_flux<D, S>(st, p, mu, pdt, divnew, prm.c, L, sg, F0, F1);
            } else {
                PwIn<D, S> dX;
                S dp, dmu;
                q1_averages<D, true>(prm, xs, xps, dX, dp, dmu);
                pw_tangent<D, S, false>(st, dX, dp, dmu, prm.c, L, sg, F0, F1);
            }
        }
        S r[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) r[f] = mul2(L.vol, q1_vgradT<D, false>(prm.fc, prm.fcr, F0[f], F1[f], (const S*)nullptr));
        chain_wait<true>();
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            T rh[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) rh[f] = half_of(r[f], h);
            const Parents P = parents_of(m, ent[h]);
            const unsigned skip0 = (skips >> (8 * h)) & 0xffu;
            if (SCAT == SCAT_WARPAGG) {
                scatter_add_warpagg<D, T>(m, out, P, rh, valid, wbuf[threadIdx.x >> 5], pin);
            } else if (SCAT == SCAT_PLAIN) {
                plain_adds<LPE>(t, valid, P.n > 1, [&] { scatter_add<D, T, SCAT_PLAIN>(m, out, P, rh, skip0, 0, pin); });
            } else if (valid) {
                scatter_add<D, T, SCAT>(m, out, P, rh, skip0, pair_rows, pin);
            }
        }
    }
}

// Threads per block of an element launch: blocks of 4 warps, or of one warp where those would
// leave SMs without a block (the FP64 pipe is per SM, so few fat blocks serialise on it).
int ek_threads(int64_t lanes) { return lanes < (int64_t)EK_THREADS * 4 * chns_num_sms() ? 32 : EK_THREADS; }

// ---------------------------------------------------------------------------------
// J^T w (reverse mode, FP64)
// ---------------------------------------------------------------------------------
template <int D, int SCAT>
__global__ void __launch_bounds__(EK_THREADS, 2)
elem_vjp_kernel(DevMesh m, const __grid_constant__ Q1Params<double> prm, double iCn, const double* __restrict__ Uo,
                const double* __restrict__ Un, const double* __restrict__ w, double* __restrict__ gn,
                double* __restrict__ go, double* __restrict__ gCn, int pin, const int32_t* __restrict__ elist,
                int64_t ecount) {
    constexpr int NC = Shape<D>::NC, NF = Shape<D>::NF;
    const int t = threadIdx.x % NC;
    const int64_t idx = (int64_t)blockIdx.x * (blockDim.x / NC) + threadIdx.x / NC;
    const bool valid = idx < ecount;
    const int64_t ie = valid ? idx : ecount - 1;
    const int64_t e = elist ? (int64_t)elist[ie] : ie;
    const PwLevel<double>& L = prm.lev[m.level[e]];
    const int ent = m.e2n[e * NC + t];
    double sg[D];
    q1_signs<D>(t, L.s, sg);
    unsigned mask;
    PwState<D, double> st;
    {
        PwIn<D, double> X;
        double gs[NF][1], gd[D + 1][1], gp[1], gx[NF][1], gxp[1], s[NF], d[D + 1], p, mu, ddiv;
        const Parents P = parents_of(m, ent);
        gather_corners<D, 1, false, double>(&P, Uo, Un, nullptr, gs, gd, gp, gx, gxp, &mask);
#pragma unroll
        for (int f = 0; f < NF; ++f) s[f] = gs[f][0];
#pragma unroll
        for (int i = 0; i <= D; ++i) d[i] = gd[i][0];
        const double ps = gp[0];
        q1_averages<D, false>(prm, s, ps, X, p, mu);
        q1_differences<D, false>(prm, sg, d, X, ddiv);
        pw_primal<D, double, false>(X, prm.c, L, sg, st);
    }
    double F0[NF], F1[NF][D];
    {
        // adjoint seed: w on rows that the element contributes to (Dirichlet and pin
        // rows are replaced rows, their element contributions are discarded)
        double sw[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) sw[f] = 0.0;
        const Parents P = parents_of(m, ent);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= P.n) break;
            const int n = parent(P, j);
            const unsigned fl = m.nflag[n];
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                double wv = __ldg(w + (size_t)n * NF + f);
                if (f < D && ((fl >> f) & 1u)) wv = 0.0;
                if (f == D && pin == 1 && n == 0) wv = 0.0;
                sw[f] = j == 0 ? wv : sw[f] + wv;
            }
        }
        const double wt = parent_weight<double>(P.n);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            double t;
            q1_vgrad<D, false>(P.n == 1 ? sw[f] : wt * sw[f], t, F1[f], (double*)nullptr);
            F0[f] = prm.fc * t;
        }
    }
    PwIn<D, double> B;
    double pb, mub, divb, cnb;
    pw_adjoint<D, double, false>(st, F0, F1, prm.c, L, sg, iCn, B, pb, mub, divb, cnb);
    // transpose of the interpolation; both levels take the averages' share, the differences +-,
    // and div v^{k+1} is div v~ plus half the difference's divergence
    double rn[NF], ro[NF];
    const double f = prm.f, fr = prm.fr;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        B.gv[i][i] = fma3(sg[i], divb, B.gv[i][i]);
        rn[i] = q1_vgradT<D, false>(f, fr, B.v[i], B.gv[i], (const double*)nullptr);
    }
    rn[D] = q1_vgradT<D, false>(prm.sp, prm.sp * Q1_R, pb, B.gp, (const double*)nullptr);
#pragma unroll
    for (int k = 0; k < Shape<D>::NH; ++k) B.H[k] *= prm.inv_f;
    rn[D + 1] = q1_vgradT<D, true>(f, fr, B.phi, B.gq, B.H);
    rn[D + 2] = q1_vgradT<D, false>(f, fr, mub, B.gm, (const double*)nullptr);
    const double psb = L.vol * q1_vgradT<D, false>(f, fr, B.ps, B.gs, (const double*)nullptr);
    double dd[D + 1];
    dd[0] = q1_vderT<D, 0>(prm.sd * B.a[0], sg[0] * divb);
    dd[1] = q1_vderT<D, 1>(prm.sd * B.a[1], sg[1] * divb);
    if constexpr (D == 3) dd[2] = q1_vderT<D, 2>(prm.sd * B.a[2], sg[2] * divb);
    {
        double b = prm.sd * B.pdt;
        if constexpr (D == 3) b = lerp(b, 4);
        dd[D] = x_lerp(lerp(b, 2));
    }
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const double a = L.vol * rn[k];
        if (k == D || k == D + 2) {
            rn[k] = ro[k] = a;
        } else {
            const double b = dd[k < D ? k : D];
            rn[k] = fma(L.vol, b, a);
            ro[k] = fma(-L.vol, b, a);
        }
    }
    chain_wait<true>();
    {
        const Parents P = parents_of(m, ent);
        const double wt = parent_weight<double>(P.n);
        const auto add = [&] {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j >= P.n) break;
                double* on = gn + (size_t)parent(P, j) * NF;
                double* oo = go ? go + (size_t)parent(P, j) * NF : nullptr;
                const double pst = (mask & (1u << j)) ? psb : 0.0;
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const double vn = wt * (f == D + 1 ? rn[f] + pst : rn[f]);
                    if (SCAT == SCAT_PLAIN) on[f] += vn;
                    else atomicAdd(on + f, vn);
                    if (oo) {
                        const double vo = wt * (f == D + 1 ? ro[f] + pst : ro[f]);
                        if (SCAT == SCAT_PLAIN) oo[f] += vo;
                        else atomicAdd(oo + f, vo);
                    }
                }
            }
        };
        if (SCAT == SCAT_PLAIN) plain_adds<NC>(t, valid, P.n > 1, add);
        else if (valid) add();
    }
    if (gCn) {
        // each Gauss point thread holds its share of d/dCn
        if (!valid) cnb = 0.0;
        cnb *= L.vol;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) cnb += __shfl_xor_sync(0xffffffffu, cnb, off);
        if ((threadIdx.x & 31) == 0 && cnb != 0.0) atomicAdd(gCn, cnb);
    }
}

template <int D, class S, int MODE>
cudaError_t launch_rj(const chns_mesh* mm, const PhysConst& pc, const typename Scalar<S>::type* Uo,
                      const typename Scalar<S>::type* Un, const typename Scalar<S>::type* x,
                      typename Scalar<S>::type* out, int pin, cudaStream_t s) {
    using T = typename Scalar<S>::type;
    constexpr int LPE = Shape<D>::NC / Lanes<S>::NP;
    const DevMesh& m = mm->dm;
    cudaError_t err = launch_init_rows<D, T, MODE>(m, MODE == MODE_RES ? Un : x, Uo, out, nullptr, nullptr, pin, s);
    if (err != cudaSuccess) return err;
    const Q1Params<S> prm = q1_params<D, S>(pc, m.hi - m.lo, mm->max_level);
    const int pair_rows = (uintptr_t)out % 8 == 0;   // the output has no alignment rule of its own
    auto grid = [&](int64_t cnt, int threads) {
        const int64_t blocks = (cnt * LPE + threads - 1) / threads;
        // FP32: two rounds of the resident blocks, each walking the elements with the indices of
        // the next ones loaded ahead (128^3: 526 us one element group per block, 478 us so; the
        // FP64 kernels wait for their pipe and take a block per group)
        const int64_t cap = sizeof(T) == 4 ? 6 * (EK_THREADS / threads) * (int64_t)chns_num_sms() : blocks;
        return (unsigned)(blocks < cap ? blocks : cap);
    };
    if (mm->scatter == SCAT_PLAIN) {
        // one launch per colour of the element colouring, fixed order: deterministic sums
        for (size_t k = 0; k + 1 < mm->colour_off.size(); ++k) {
            const int64_t c0 = mm->colour_off[k], cnt = mm->colour_off[k + 1] - c0;
            if (cnt <= 0) continue;
            const int th = ek_threads(cnt * LPE);
            elem_rj_kernel<D, S, MODE, SCAT_PLAIN><<<grid(cnt, th), th, 0, s>>>(
                m, prm, Uo, Un, x, out, mm->d_flags, mm->d_elist + c0, cnt, 0, pin);
            chns_count_launches(1);
        }
    } else {
        const int th = ek_threads(m.E * LPE);
        if (mm->scatter == SCAT_WARPAGG)
            chain<true>(elem_rj_kernel<D, S, MODE, SCAT_WARPAGG>, grid(m.E, th), th, s,
                m, prm, Uo, Un, x, out, mm->d_flags, nullptr, m.E, 0, pin);
        else
            chain<true>(elem_rj_kernel<D, S, MODE, SCAT_ATOMIC>, grid(m.E, th), th, s,
                m, prm, Uo, Un, x, out, mm->d_flags, nullptr, m.E, pair_rows, pin);
        chns_count_launches(1);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_residual(const chns_mesh* m, const PhysConst& pc, const double* U_old, const double* U_new,
                            double* R, int pin, cudaStream_t s) {
    if (m->dm.dim == 2) return launch_rj<2, double, MODE_RES>(m, pc, U_old, U_new, nullptr, R, pin, s);
    return launch_rj<3, double, MODE_RES>(m, pc, U_old, U_new, nullptr, R, pin, s);
}

cudaError_t launch_jvp64(const chns_mesh* m, const PhysConst& pc, const double* U_old, const double* U_lin,
                         const double* x, double* y, int pin, cudaStream_t s) {
    if (m->dm.dim == 2) return launch_rj<2, double, MODE_JVP>(m, pc, U_old, U_lin, x, y, pin, s);
    return launch_rj<3, double, MODE_JVP>(m, pc, U_old, U_lin, x, y, pin, s);
}

cudaError_t launch_jvp32(const chns_mesh* m, const PhysConst& pc, const float* U_old, const float* U_lin,
                         const float* x, float* y, int pin, cudaStream_t s) {
    if (m->dm.dim == 2) return launch_rj<2, float2, MODE_JVP>(m, pc, U_old, U_lin, x, y, pin, s);
    return launch_rj<3, float2, MODE_JVP>(m, pc, U_old, U_lin, x, y, pin, s);
}

cudaError_t launch_vjp(const chns_mesh* mm, const PhysConst& pc, const double* U_old, const double* U_lin,
                       const double* w, double* gU_new, double* gU_old, double* gCn, int pin, cudaStream_t s) {
    const DevMesh& m = mm->dm;
    auto elems = [&](auto dimtag) -> cudaError_t {
        constexpr int D = decltype(dimtag)::value, NC = Shape<D>::NC;
        const cudaError_t err = launch_init_rows<D, double, ROWS_VJP>(m, w, nullptr, gU_new, gU_old, gCn, pin, s);
        if (err != cudaSuccess) return err;
        const Q1Params<double> prm = q1_params<D, double>(pc, m.hi - m.lo, mm->max_level);
        if (mm->scatter == SCAT_PLAIN) {
            for (size_t k = 0; k + 1 < mm->colour_off.size(); ++k) {
                const int64_t c0 = mm->colour_off[k], cnt = mm->colour_off[k + 1] - c0;
                if (cnt <= 0) continue;
                const int th = ek_threads(cnt * NC);
                elem_vjp_kernel<D, SCAT_PLAIN><<<(unsigned)((cnt * NC + th - 1) / th), th, 0, s>>>(
                    m, prm, 1.0 / pc.Cn, U_old, U_lin, w, gU_new, gU_old, gCn, pin, mm->d_elist + c0, cnt);
                chns_count_launches(1);
            }
        } else {
            const int th = ek_threads(m.E * NC);
            chain<true>(elem_vjp_kernel<D, SCAT_ATOMIC>, (unsigned)((m.E * NC + th - 1) / th), th, s,
                m, prm, 1.0 / pc.Cn, U_old, U_lin, w, gU_new, gU_old, gCn, pin, nullptr, m.E);
            chns_count_launches(1);
        }
        return cudaGetLastError();
    };
    return m.dim == 2 ? elems(std::integral_constant<int, 2>()) : elems(std::integral_constant<int, 3>());
}
