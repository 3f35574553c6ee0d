// Rows that the boundary conditions replace: Dirichlet velocity components and the pinned pressure.
#pragma once

#include <cuda_runtime.h>

#include "chain.cuh"
#include "chns_internal.h"

namespace {

// bit f < D: velocity component f of the node is a Dirichlet row; bit D: its pressure is pinned
template <int D>
__device__ __forceinline__ unsigned replaced_rows(const DevMesh& m, int node, int pin) {
    unsigned fl = __ldg(m.nflag + node) & ((1u << D) - 1u);
    if (pin == 1 && node == 0) fl |= 1u << D;
    return fl;
}

// Clears the output and writes the replaced rows (Dirichlet velocity components, pressure pin):
//   residual: R = v^{k+1} - g on the Dirichlet rows (g: prescribed velocity, zero when the
//             mesh has none); R[0,p] = p^{k+1} - p^k
//   J x     : y = x on those rows
//   J^T w   : g_new = w on those rows, to which the elements add; g_old = -w at the pin
// One pass in the place of a memset before the elements and a boundary kernel after them: a
// call is two launches instead of three (five for J^T w), 4 us less of a small call's 23.  The
// element kernel starts beside it (chain.cuh) and waits for it only where it adds to the output
// (64^3 FP32 J x: 73 to 69 us; 32^2 FP64: 18.5 to 16.5 us).
enum { ROWS_RES = 0, ROWS_JVP = 1, ROWS_VJP = 2 };
template <int D, class T, int MODE>
__global__ void __launch_bounds__(256) init_rows_kernel(DevMesh m, const T* __restrict__ a, const T* __restrict__ b, T* __restrict__ out,
                                 T* __restrict__ out_old, T* __restrict__ gCn, int pin) {
    constexpr int NF = (D + 3);
    chain_next<true>();
    // a block covers 256 nodes, entry by entry
    const int64_t node0 = (int64_t)blockIdx.x * 256;
    T* const o = out + node0 * NF;
    const T* const ai = a + node0 * NF;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const unsigned j = k * 256u + threadIdx.x, nl = j / NF;
        const int f = (int)(j - nl * NF);
        const int64_t node = node0 + nl;
        if (node >= m.N) break;
        T v = T(0), vo = T(0);
        if (f < D && ((__ldg(m.nflag + node) >> f) & 1u)) {
            v = ai[j];
            if (MODE == ROWS_RES && m.bcval) v -= (T)m.bcval[node * D + f];
        }
        if (pin == 1 && node == 0 && f == D) {
            v = MODE == ROWS_RES ? ai[j] - b[j] : ai[j];
            vo = -ai[j];
        }
        o[j] = v;
        if (MODE == ROWS_VJP && out_old) out_old[node0 * NF + j] = vo;
    }
    if (MODE == ROWS_VJP && gCn && blockIdx.x == 0 && threadIdx.x == 0) gCn[0] = T(0);
}
template <int D, class T, int MODE>
cudaError_t launch_init_rows(const DevMesh& m, const T* a, const T* b, T* out, T* out_old, T* gCn, int pin,
                             cudaStream_t s) {
    init_rows_kernel<D, T, MODE><<<(unsigned)((m.N + 255) / 256), 256, 0, s>>>(m, a, b, out, out_old, gCn, pin);
    chns_count_launches(1);
    return cudaGetLastError();
}

}  // namespace
