// Reductions of the hot path in FP64: mass (integral of phi, Proposition 1), the parts of
// the energy functional (Eq. energy_functional), and the BLAS-1 building blocks of the
// Krylov solver.  Every reduction is deterministic: a fixed grid writes one partial per
// block (warp shuffles, then shared memory), and one block sums the partials in a fixed order
// (the last one to finish; the dot products: a second kernel).
#include <cuda_runtime.h>

#include "chns_internal.h"
#include "krylov.h"
#include "q1_lanes.cuh"
#include "reduce.cuh"

namespace {

constexpr int RT = 256;

// int phi = sum_n m_n phi_n (m_n: the integral of node n's basis function, hanging weights included)
__global__ void __launch_bounds__(RT) mass_kernel(const double* __restrict__ mass, const double* __restrict__ U, int NF, int f,
                                                  int64_t N, double* partials, unsigned int* counter, double* out) {
    double acc[1] = {0.0};
    for (int64_t n = (int64_t)blockIdx.x * RT + threadIdx.x; n < N; n += (int64_t)gridDim.x * RT)
        acc[0] = fma(mass[n], U[(size_t)n * NF + f], acc[0]);
    block_reduce_store<1>(acc, partials);
    if (!krylov::last_block(counter) || threadIdx.x >= 32) return;
    double v = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) v += __ldcg(partials + b);
    v = krylov::warp_sum(v);
    if (threadIdx.x == 0) out[0] = v;
}

// The three parts of the energy, a lane per Gauss point (the exchange of q1_lanes.cuh: about 45 FP64
// operations per point, where summing basis products took 230; 165,824 elements: 290 -> 171 us)
template <int D>
__global__ void __launch_bounds__(RT) energy_kernel(DevMesh m, double alpha, double beta, double Cn, double inv_CnWe, double inv_Fr,
                                                    const double* __restrict__ U, double* partials, unsigned int* counter,
                                                    double* out) {
    constexpr int NC = Shape<D>::NC, NF = Shape<D>::NF;
    constexpr double f = D == 2 ? Q1_CP * Q1_CP : Q1_CP * Q1_CP * Q1_CP;
    const double L = m.hi - m.lo, unit = L * pow2(-m.max_level), detL = D == 2 ? 0.25 * L * L : 0.125 * L * L * L;
    const double s0 = Cn * f / (L * Q1_CP), g0 = 0.5 * s0 * s0;
    const int t = threadIdx.x % NC;
    double acc[3] = {0.0, 0.0, 0.0};
    for (int64_t base = (int64_t)blockIdx.x * (RT / NC); base < m.E; base += (int64_t)gridDim.x * (RT / NC)) {
        const int64_t idx = base + threadIdx.x / NC;
        const bool valid = idx < m.E;
        const int64_t e = valid ? idx : m.E - 1;
        const Parents P = parents_of(m, __ldg(m.e2n + e * NC + t));
        // v, phi, phi* (clip at independent nodes)
        double u[D + 2];
#pragma unroll
        for (int k = 0; k < D + 2; ++k) u[k] = 0.0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= P.n) break;
            const double* r = U + (size_t)parent(P, j) * NF;
#pragma unroll
            for (int k = 0; k < D; ++k) u[k] = j == 0 ? __ldg(r + k) : u[k] + __ldg(r + k);
            const double phi = __ldg(r + D + 1), ps = fmin(1.0, fmax(-1.0, phi));
            u[D] = j == 0 ? phi : u[D] + phi;
            u[D + 1] = j == 0 ? ps : u[D + 1] + ps;
        }
        if (P.n > 1) {
            const double w = parent_weight<double>(P.n);
#pragma unroll
            for (int k = 0; k < D + 2; ++k) u[k] *= w;
        }
        double vv = 0.0, phi, g[D], gg = 0.0;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            const double v = q1_value<D>(u[k]);
            vv = fma(v, v, vv);
        }
        q1_vgrad<D, false>(u[D], phi, g, (double*)nullptr);
        phi *= f;
#pragma unroll
        for (int k = 0; k < D; ++k) gg = fma(g[k], g[k], gg);
        const double rho = fma(alpha * f, q1_value<D>(u[D + 1]), beta);
        const int lev = m.level[e];
        const double detJ = valid ? detL * pow2(-D * lev) : 0.0;
        const double q = fma(phi, phi, -1.0);
        acc[0] = fma(detJ * (0.5 * f * f), rho * vv, acc[0]);
        acc[1] = fma(detJ, fma(0.25 * q, q, g0 * pow2(2 * lev) * gg), acc[1]);
        if (inv_Fr != 0.0) {
            const double z = m.lo + unit * (double)m.anchor[e * D + D - 1] + L * pow2(-lev) * (((t >> (D - 1)) & 1) ? Q1_CP : 1.0 - Q1_CP);
            acc[2] = fma(detJ * rho, z, acc[2]);
        }
    }
    acc[1] *= inv_CnWe;
    acc[2] *= inv_Fr;
    block_reduce_store<3>(acc, partials);
    if (!krylov::last_block(counter) || threadIdx.x >= 96) return;
    const int k = threadIdx.x >> 5;
    double v = 0.0;
    for (int b = threadIdx.x & 31; b < (int)gridDim.x; b += 32) v += __ldcg(partials + (size_t)b * 3 + k);
    v = krylov::warp_sum(v);
    if ((threadIdx.x & 31) == 0) out[k] = v;
}

template <int K>
__global__ void dot_kernel(const double* __restrict__ a, const double* __restrict__ b, int64_t n,
                           double* partials) {
    double acc[1] = {0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        acc[0] += a[i] * b[i];
    block_reduce_store<1>(acc, partials);
}

int reduce_blocks(int64_t work) {
    int64_t b = (work + 255) / 256;
    const int64_t cap = 4 * (int64_t)chns_num_sms();
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

}  // namespace

__global__ void final_reduce_kernel(const double* __restrict__ partials, int nblocks, int K,
                                    double* __restrict__ out) {
    __shared__ double sh[256];
    for (int k = 0; k < K; ++k) {
        double v = 0.0;
        for (int i = threadIdx.x; i < nblocks; i += blockDim.x) v += partials[(size_t)i * K + k];
        sh[threadIdx.x] = v;
        __syncthreads();
        for (int s = 128; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0) out[k] = sh[0];
        __syncthreads();
    }
}

cudaError_t launch_mass(const chns_mesh* mm, const double* U, double* out_dev, cudaStream_t s) {
    const DevMesh& m = mm->dm;
    mass_kernel<<<reduce_blocks(m.N), RT, 0, s>>>(mm->d_nmass, U, m.nf, m.dim + 1, m.N, mm->d_partials, mm->d_flags + 8, out_dev);
    chns_count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_energy(const chns_mesh* mm, const PhysConst& pc, const double* U, double* out_dev3,
                          cudaStream_t s) {
    const DevMesh& m = mm->dm;
    const int nb = reduce_blocks(m.E * m.nc);
    const double inv_CnWe = 1.0 / (pc.Cn * pc.We);
    if (m.dim == 2)
        energy_kernel<2><<<nb, RT, 0, s>>>(m, pc.alpha, pc.beta, pc.Cn, inv_CnWe, pc.inv_Fr, U, mm->d_partials, mm->d_flags + 8, out_dev3);
    else
        energy_kernel<3><<<nb, RT, 0, s>>>(m, pc.alpha, pc.beta, pc.Cn, inv_CnWe, pc.inv_Fr, U, mm->d_partials, mm->d_flags + 8, out_dev3);
    chns_count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_dot(const chns_mesh* mm, const double* a, const double* b, int64_t n, double* out_dev,
                       cudaStream_t s) {
    const int nb = reduce_blocks(n);
    { dot_kernel<1><<<nb, 256, 0, s>>>(a, b, n, mm->d_partials); chns_count_launches(1); }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    { final_reduce_kernel<<<1, 256, 0, s>>>(mm->d_partials, nb, 1, out_dev); chns_count_launches(1); }
    return cudaGetLastError();
}
