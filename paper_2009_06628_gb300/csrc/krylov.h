// Arnoldi vectors of Newton's GMRES and the adjoint's (krylov.cu).
#pragma once

#include <cuda_runtime.h>

#include "chns_internal.h"

// device scalars (indices into SolverWS::sc)
enum {
    SC_H1 = 0,          // first-pass coefficients
    SC_H2 = 256,        // second-pass coefficients
    SC_NB = 600,        // |w|^2 before the first pass
    SC_NA = 603,        // |w|^2 after the last pass
    SC_AGAIN = 605,     // 1: a second pass runs
    SC_MEAN = 610,      // m_p^T z
    SC_SCALE = 640,     // s_j, j <= 256
    SC_MISC = 900
};

namespace krylov {

constexpr int T = 256;          // threads per block
constexpr int COLUMNS = 256;    // at most
constexpr int COUNTERS = 32;    // one per chunk of columns

// sum over the warp, in every lane (all 32 call it)
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// true in every thread of the block that finished last
__device__ __forceinline__ bool last_block(unsigned int* counter) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int t = atomicAdd(counter, 1u);
        last = t == gridDim.x - 1;
        if (last) *counter = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

// w_i = S_i y_i (+ mean on the rows of field f): the operator's result, formed where it is read
struct Source {
    const float* yf;        // the result, in FP32 or FP64 (both null: w is in place)
    const double* yd;
    const double* S;
    const double* mean;     // null: none
    double a;
    int NF, f;
};

// Gram-Schmidt of w (slot k of V, or formed there from src) against slots 0..k-1: coefficients,
// norms and s_k in sc; host (pinned) gets the coefficients of both passes together in [0, k) and
// |w|^2 in [SC_NA].  thr: re-orthogonalise when |w|^2 falls below thr times its old value (infinity:
// always).  One launch for short vectors with few columns, else four, and two more per 32 columns beyond
// 32 for long ones; returns their number.
// partials: 33 doubles for each of 4 blocks per SM (of 8 SMs at least); counter: COUNTERS words, zero.
int orthogonalise(double* V, int64_t ld, int k, const Source& src, int64_t n, double* sc, double thr, double* host, double* partials,
                  unsigned int* counter, cudaStream_t st);
// u = sum_{j<k} y_j v_j
void combine(const double* V, int64_t ld, int k, const double* y, const double* scale, double* u, int64_t n, cudaStream_t st);

}  // namespace krylov
