// The consistent Q1 mass matrix: the discrete initial chemical potential M mu = b(phi) and plain
// solves M x = rhs, by preconditioned conjugate gradients to a relative residual of 1e-14 (FP64,
// hanging constraints included).
//
// M is applied element by element: on a cube it is the tensor product of (h/6)(2 1; 1 2), so with
// one lane per corner each axis costs one multiply-add with the neighbour's value, 6 operations per
// corner in all (forming the basis at every Gauss point took about 150, on the FP64 pipe that
// bounded it).
//
// The preconditioner is the sum of the elements' own inverses, weighted by the nodes' masses,
//     D^-1 [ sum_e R_e^T (D_e M_e^-1 D_e) R_e ] D^-1,   D_e = (h/2)^d I,  D = sum_e R_e^T D_e 1 = m,
// and D_e M_e^-1 D_e is again a tensor product, of (h/2)(2 -1; -1 2): the same kernel with other
// signs.  On a uniform mesh the 1D symbol of the product is (4 - cos^2)/3, so the condition number
// is at most (4/3)^d, 2.4 in 3D, where the diagonal leaves 27: a third of the iterations, each with
// two passes over the elements in place of one.
//
// An iteration is three kernels: the preconditioner (r.z), the matrix (which forms p where it
// gathers it; p.q), and the nodes (all vector updates, r.r).  The last block of each turns the sums
// into beta, alpha and the stop flag, so the host only looks every few iterations, one batch
// behind; kernels behind the last iteration return at once.
//   165,824 elements with hanging corners: preconditioner 31, matrix 43, nodes 8 us, 33 iterations; a
//   solve takes 3.1 ms (Jacobi with this element kernel, 80 iterations: 5.8 ms; Gauss-point mass
//   kernel, three dots, five vector kernels and three host round trips per iteration: 13.2 ms).
//   FP64 units 80 % busy in the matrix kernel: a warp with one hanging corner runs its branch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "chns_internal.h"
#include "krylov.h"
#include "q1_lanes.cuh"

struct MassWS {
    double* v = nullptr;              // y, r, z, p, q, x, 1 / mass: N each
    double* sc = nullptr;             // device scalars (below)
    double* part = nullptr;           // block partials
    unsigned int* counter = nullptr;
    double* host = nullptr;           // pinned, two sets of scalars
    cudaEvent_t ev[2] = {};
};

namespace {

enum { CG_RZ, CG_ALPHA, CG_BETA, CG_TOL, CG_DONE, CG_ITS, CG_N };   // CG_DONE: 1 converged, 2 not finite
constexpr int CG_T = 256, CG_BATCH = 4, CG_MAX = 1000;

// sum over the block (CG_T threads) in thread 0
__device__ __forceinline__ double block_sum(double v, double* sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    v = 0.0;
    if (threadIdx.x < 32) {
#pragma unroll
        for (int q = 0; q < CG_T / 32; ++q) v += sh[threadIdx.x + 32 * q];
        v = krylov::warp_sum(v);
    }
    __syncthreads();
    return v;
}

// b_a = sum_q |J| (N_a psi'(phi_q) + Cn^2 grad N_a . grad phi_q), added into y.  c0 and detf: the
// scale of the gradient terms (Cn^2 f / (h c_+)^2) and |J| f at h = the box, powers of two apart
// from an element's
template <int D>
__global__ void __launch_bounds__(CG_T) mu_rhs_kernel(DevMesh m, double c0, double detf, const double* __restrict__ U, double* __restrict__ y) {
    constexpr int NC = Shape<D>::NC, NF = Shape<D>::NF;
    constexpr double f = D == 2 ? Q1_CP * Q1_CP : Q1_CP * Q1_CP * Q1_CP;   // value scale of the exchange
    const int t = threadIdx.x % NC;
    const int64_t idx = (int64_t)blockIdx.x * (CG_T / NC) + threadIdx.x / NC;
    const bool valid = idx < m.E;
    const int64_t e = valid ? idx : m.E - 1;
    const Parents P = parents_of(m, __ldg(m.e2n + e * NC + t));
    double u = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (j < P.n) u += __ldg(U + (size_t)parent(P, j) * NF + D + 1);
    const double w = parent_weight<double>(P.n);
    u *= w;
    double phi, g[D];
    q1_vgrad<D, false>(u, phi, g, (double*)nullptr);
    phi *= f;
    const int lev = m.level[e];
    // gradients of the exchange carry f/(h c_+) = s: d_k u d_k N_a = s^2 g_k (exchange of N_a)_k
    const double c = c0 * pow2(2 * lev);
#pragma unroll
    for (int k = 0; k < D; ++k) g[k] *= c;
    const double r = detf * pow2(-D * lev) * q1_vgradT<D, false>(1.0, Q1_R, fma(phi * phi, phi, -phi), g, (const double*)nullptr);
    if (valid)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < P.n) atomicAdd(y + parent(P, j), w * r);
}

// the last block: sums of the K partials per block of a grid, in thread 0
template <int K>
__device__ __forceinline__ void grid_sums(double* v, const double* part, double* sh) {
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += CG_T)
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] += __ldcg(part + K * b + k);
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = block_sum(v[k], sh);
}

// r given: y = D^-1 r, x = z = p = q = 0, |r| and the stopping tolerance
__global__ void __launch_bounds__(CG_T) cg_start_kernel(int64_t N, const double* __restrict__ mass, const double* __restrict__ r,
                                                        double* __restrict__ y, double* __restrict__ z, double* __restrict__ p,
                                                        double* __restrict__ q, double* __restrict__ x, double* __restrict__ dinv,
                                                        double* __restrict__ sc, double* __restrict__ part,
                                                        unsigned int* counter) {
    __shared__ double sh[CG_T];
    double rr = 0.0;
    for (int64_t n = (int64_t)blockIdx.x * CG_T + threadIdx.x; n < N; n += (int64_t)gridDim.x * CG_T) {
        const double rn = r[n], d = 1.0 / mass[n];
        dinv[n] = d;
        y[n] = d * rn;
        z[n] = p[n] = q[n] = x[n] = 0.0;
        rr = fma(rn, rn, rr);
    }
    rr = block_sum(rr, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = rr;
    if (!krylov::last_block(counter)) return;
    grid_sums<1>(&rr, part, sh);
    if (threadIdx.x == 0) {
        sc[CG_RZ] = 0.0;
        sc[CG_TOL] = 1e-14 * sqrt(rr);
        sc[CG_DONE] = rr > 0.0 ? 0.0 : 1.0;   // a right-hand side without a norm (zero, NaN): x = 0
        sc[CG_ITS] = 0.0;
    }
}

// PC: z += [sum_e R_e^T (D_e M_e^-1 D_e) R_e] y; r.z (= y . the sum), beta.
// else q += M p with p = D^-1 z + beta p formed at the corners; alpha = r.z / p.q
template <int D, bool PC>
__global__ void __launch_bounds__(CG_T) cg_element_kernel(DevMesh m, const double* __restrict__ dinv, const double* __restrict__ z,
                                                          const double* __restrict__ p, double* __restrict__ out,
                                                          double* __restrict__ sc, double* __restrict__ part, unsigned int* counter) {
    constexpr int NC = Shape<D>::NC;
    __shared__ double sh[CG_T];
    if (sc[CG_DONE] != 0.0) return;
    const double beta = sc[CG_BETA], h0 = (m.hi - m.lo) / (PC ? 2.0 : 6.0), s0 = D == 2 ? h0 * h0 : h0 * h0 * h0;
    const int t = threadIdx.x % NC;
    const auto at = [&](int n) { return PC ? __ldg(z + n) : fma(beta, __ldg(p + n), __ldg(dinv + n) * __ldg(z + n)); };
    double ua = 0.0;
    for (int64_t base = (int64_t)blockIdx.x * (CG_T / NC); base < m.E; base += (int64_t)gridDim.x * (CG_T / NC)) {
        const int64_t idx = base + threadIdx.x / NC;
        const bool valid = idx < m.E;
        const int64_t e = valid ? idx : m.E - 1;
        const Parents P = parents_of(m, __ldg(m.e2n + e * NC + t));
        double u = at(P.p.x);
        const double w = parent_weight<double>(P.n);
        if (P.n > 1) {
#pragma unroll
            for (int j = 1; j < 4; ++j)
                if (j < P.n) u += at(parent(P, j));
            u *= w;
        }
        constexpr double c = PC ? -2.0 : 2.0;   // +-(2 -+1; -+1 2) per axis; the sign comes out below
        double a = fma(c, u, shx(u, 1));
        a = fma(c, a, shx(a, 2));
        if constexpr (D == 3) a = fma(c, a, shx(a, 4));
        a *= (PC && D == 3 ? -s0 : s0) * pow2(-D * (int)m.level[e]);
        if (valid) {
            ua = fma(u, a, ua);
            if (P.n == 1) {
                atomicAdd(out + P.p.x, a);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (j < P.n) atomicAdd(out + parent(P, j), w * a);
            }
        }
    }
    ua = block_sum(ua, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = ua;
    if (!krylov::last_block(counter)) return;
    grid_sums<1>(&ua, part, sh);
    if (threadIdx.x == 0) {
        const double rz = sc[CG_RZ];
        if (PC) {
            sc[CG_BETA] = rz > 0.0 ? ua / rz : 0.0;
            sc[CG_RZ] = ua;
        } else {
            sc[CG_ALPHA] = rz / ua;
        }
    }
}

// p = D^-1 z + beta p, x += alpha p, r -= alpha q, y = D^-1 r, z = q = 0; the stop flag
__global__ void __launch_bounds__(CG_T) cg_update_kernel(int64_t N, const double* __restrict__ dinv, double* __restrict__ r,
                                                         double* __restrict__ y, double* __restrict__ z, double* __restrict__ p,
                                                         double* __restrict__ q, double* __restrict__ x, double* __restrict__ sc,
                                                         double* __restrict__ part, unsigned int* counter) {
    __shared__ double sh[CG_T];
    if (sc[CG_DONE] != 0.0) return;
    const double alpha = sc[CG_ALPHA], beta = sc[CG_BETA];
    double rr = 0.0;
    for (int64_t n = (int64_t)blockIdx.x * CG_T + threadIdx.x; n < N; n += (int64_t)gridDim.x * CG_T) {
        const double d = dinv[n], pn = fma(beta, p[n], d * z[n]), rn = fma(-alpha, q[n], r[n]);
        p[n] = pn;
        x[n] = fma(alpha, pn, x[n]);
        r[n] = rn;
        y[n] = d * rn;
        z[n] = q[n] = 0.0;
        rr = fma(rn, rn, rr);
    }
    rr = block_sum(rr, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = rr;
    if (!krylov::last_block(counter)) return;
    grid_sums<1>(&rr, part, sh);
    if (threadIdx.x == 0) {
        sc[CG_ITS] += 1.0;
        if (!(rr <= 1.7e308)) sc[CG_DONE] = 2.0;
        else if (sqrt(rr) <= sc[CG_TOL]) sc[CG_DONE] = 1.0;
    }
}

__global__ void insert_field_kernel(const double* __restrict__ in, int NF, int f, int64_t N, double* __restrict__ U) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n < N) U[(size_t)n * NF + f] = in[n];
}

chns_status ensure_mass_ws(chns_mesh* m) {
    if (m->mass) return CHNS_OK;
    MassWS* w = new (std::nothrow) MassWS();
    if (!w) { chns_set_error("host allocation failed"); return CHNS_ENOMEM; }
    cudaError_t e = cudaMalloc((void**)&w->v, (size_t)7 * m->dm.N * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&w->sc, CG_N * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&w->part, (size_t)2 * 8 * chns_num_sms() * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&w->counter, sizeof(unsigned int));
    if (e == cudaSuccess) e = cudaMemset(w->counter, 0, sizeof(unsigned int));
    if (e == cudaSuccess) e = cudaMallocHost((void**)&w->host, 2 * CG_N * sizeof(double));
    for (auto& ev : w->ev)
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        chns_mass_ws_free(w);
        return chns_cuda_status(e, "cudaMalloc(mass solve workspace)");
    }
    m->mass = w;
    return CHNS_OK;
}

// M x = r (r is overwritten; both in the workspace or the caller's)
chns_status cg_solve(chns_mesh* m, double* r, double* x, cudaStream_t s) {
    MassWS* w = m->mass;
    const int64_t N = m->dm.N;
    double *y = w->v, *z = w->v + 2 * N, *p = w->v + 3 * N, *q = w->v + 4 * N, *dinv = w->v + 6 * N;
    const int64_t sms = chns_num_sms();
    const int gn = (int)std::min<int64_t>((N + CG_T - 1) / CG_T, 8 * sms);
    const int ge = (int)std::min<int64_t>((m->dm.E * m->dm.nc + CG_T - 1) / CG_T, 8 * sms);
    const auto elements = m->dm.dim == 2 ? cg_element_kernel<2, false> : cg_element_kernel<3, false>;
    const auto inverses = m->dm.dim == 2 ? cg_element_kernel<2, true> : cg_element_kernel<3, true>;
    cg_start_kernel<<<gn, CG_T, 0, s>>>(N, m->d_nmass, r, y, z, p, q, x, dinv, w->sc, w->part, w->counter);
    chns_count_launches(1);
    CHNS_CUDA(cudaGetLastError());
    for (int batch = 0;; ++batch) {
        // one batch is queued ahead of the one whose flag the host waits for
        const bool more = batch * CG_BATCH < CG_MAX;
        if (more) {
            for (int i = 0; i < CG_BATCH; ++i) {
                inverses<<<ge, CG_T, 0, s>>>(m->dm, nullptr, y, nullptr, z, w->sc, w->part, w->counter);
                elements<<<ge, CG_T, 0, s>>>(m->dm, dinv, z, p, q, w->sc, w->part, w->counter);
                cg_update_kernel<<<gn, CG_T, 0, s>>>(N, dinv, r, y, z, p, q, x, w->sc, w->part, w->counter);
            }
            chns_count_launches(3 * CG_BATCH);
            CHNS_CUDA(cudaGetLastError());
            CHNS_CUDA(cudaMemcpyAsync(w->host + (batch & 1) * CG_N, w->sc, CG_N * sizeof(double), cudaMemcpyDeviceToHost, s));
            CHNS_CUDA(cudaEventRecord(w->ev[batch & 1], s));
        }
        if (batch == 0) continue;
        CHNS_CUDA(cudaEventSynchronize(w->ev[(batch - 1) & 1]));
        const double* h = w->host + ((batch - 1) & 1) * CG_N;
        if (h[CG_DONE] != 0.0) CHNS_CUDA(cudaStreamSynchronize(s));   // the batch behind it
        if (h[CG_DONE] == 2.0) { chns_set_error("non-finite CG residual"); return CHNS_ENAN; }
        if (h[CG_DONE] == 1.0) return CHNS_OK;
        if (!more) { chns_set_error("mass-matrix CG did not converge"); return CHNS_ENOCONV; }
    }
}

}  // namespace

void chns_mass_ws_free(MassWS* w) {
    if (!w) return;
    cudaFree(w->v);
    cudaFree(w->sc);
    cudaFree(w->part);
    cudaFree(w->counter);
    if (w->host) cudaFreeHost(w->host);
    for (auto& e : w->ev)
        if (e) cudaEventDestroy(e);
    delete w;
}

extern "C" chns_status chns_initial_mu(const chns_mesh* mc, const chns_params* p, double* U, void* stream) {
    if (chns_require_q1(mc, "chns_initial_mu") != CHNS_OK) return CHNS_EINVAL;
    chns_mesh* m = const_cast<chns_mesh*>(mc);
    PhysConst pc;
    chns_status st = chns_check_params(mc, p, &pc);
    if (st != CHNS_OK) return st;
    if (!U) { chns_set_error("null argument"); return CHNS_EINVAL; }
    if ((st = ensure_mass_ws(m)) != CHNS_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t N = m->dm.N;
    const int D = m->dm.dim, NF = m->dm.nf;
    double *r = m->mass->v + N, *x = m->mass->v + 5 * N;
    CHNS_CUDA(cudaMemsetAsync(r, 0, N * sizeof(double), s));
    const unsigned ge = (unsigned)((m->dm.E * m->dm.nc + CG_T - 1) / CG_T);
    const double L = m->dm.hi - m->dm.lo, f = std::pow(Q1_CP, D);
    const double c0 = p->Cn * p->Cn * f / (L * L * (Q1_CP * Q1_CP)), detf = std::pow(0.5 * L, D) * f;
    if (D == 2) mu_rhs_kernel<2><<<ge, CG_T, 0, s>>>(m->dm, c0, detf, U, r);
    else mu_rhs_kernel<3><<<ge, CG_T, 0, s>>>(m->dm, c0, detf, U, r);
    chns_count_launches(1);
    CHNS_CUDA(cudaGetLastError());
    st = cg_solve(m, r, x, s);
    // a solve that ran out of iterations leaves its last iterate; one that is not finite, nothing
    if (st == CHNS_OK || st == CHNS_ENOCONV) {
        insert_field_kernel<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(x, NF, D + 2, N, U);
        chns_count_launches(1);
        CHNS_CUDA(cudaGetLastError());
        CHNS_CUDA(cudaStreamSynchronize(s));
    }
    return st;
}

// M x = rhs (M is symmetric, so its adjoint is the same solve); used by the reverse mode of mu^0.
extern "C" chns_status chns_mass_solve(const chns_mesh* mc, const double* rhs, double* x, void* stream) {
    if (chns_require_q1(mc, "chns_mass_solve") != CHNS_OK) return CHNS_EINVAL;
    chns_mesh* m = const_cast<chns_mesh*>(mc);
    if (!m || !rhs || !x) { chns_set_error("null argument"); return CHNS_EINVAL; }
    chns_status st = ensure_mass_ws(m);
    if (st != CHNS_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    double* r = m->mass->v + m->dm.N;
    CHNS_CUDA(cudaMemcpyAsync(r, rhs, m->dm.N * sizeof(double), cudaMemcpyDeviceToDevice, s));
    st = cg_solve(m, r, x, s);
    CHNS_CUDA(cudaStreamSynchronize(s));
    return st;
}
