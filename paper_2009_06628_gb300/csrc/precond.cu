// Assembled scalar Q1 operators and the preconditioners built on them: the pressure
// Schur-complement approximation (grad q, dt/(2 rho We) grad p), inverted by a
// Jacobi-preconditioned Chebyshev polynomial or one geometric multigrid V-cycle, and the
// Cahn-Hilliard block (M + eps K) M^{-1} (M + eps K), eps^2 = dt Cn/(2 Pe).  FP32.
//
// Why assembled.  These operators are applied 15 to 70 times per preconditioner application to
// one vector that fits in L2, so the time is the length of a chain of short kernels, not their
// arithmetic.  Element-wise, a step was two kernels (8 gathers and 8 atomics per element into a
// zeroed vector, then the vector update that the atomics have to wait for).  With rows, one
// kernel gathers, reduces and updates: half the chain, no atomics, a fixed summation order.
//   64^3 (274,625 rows), degree 16: a whole preconditioner application 313 -> 125 us (15 of them the
//   block-Jacobi part); 45,000 rows with hanging points, V-cycle and Cahn-Hilliard block: 620 -> 140
//   us; 1,089 rows in 2D, degree 16: 90 -> 25 us.
// Rows are stored in slices of 32 (one warp), column-major within a slice and padded to its
// longest row, so that every load of columns and values is one full line; rows next to each
// other in Morton order have near-equal lengths.  With hanging nodes a row also holds the
// columns that the constraints fold in.  The pressure operator drops the couplings along an
// element edge, whose stiffness entry on a cube is zero (21 of 27 columns remain in 3D).
//
// Levels whose matrix is small run in one block, a block barrier per phase instead of a launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <type_traits>
#include <utility>
#include <vector>

#include "chain.cuh"
#include "precond.h"

namespace {

constexpr int MAX_DEG = 200;
constexpr int CH_DEG = 8;
constexpr int COARSE_DEG = 16;
constexpr int TAIL_THREADS = 1024;
constexpr int TAIL_ROWS = 2 * TAIL_THREADS;
// Levels of the one-block kernel: those whose matrix its registers hold, from degree 5 on, and those
// with so few entries that a step through L1 costs no more than a launched one.  A launched step is
// 1.5 us at these sizes and one from registers 0.8; through L1 it is 1.5 at 2,601 entries and 6.4 at 38,025.
//   Polynomial, degree 16, us per application, launched / here (block-Jacobi part included): 289 rows in 2D
//   33 / 19, 1,089 rows 34 / 25, 729 rows in 3D 36 / 27; through L1: 2,681 rows in 2D with hanging points 34 / 88,
//   4,225 rows 34 / 112, 1,049 rows in 3D with hanging points 50 / 96.
//   V-cycle, degree 2, with all levels of up to 40,960 / 20,480 / 10,240 / 5,120 / 0 entries here: 66,049 rows in
//   2D 122 / 89 / 89 / 81 / 81 us, 1,497 rows (hanging) 58 / 58 / 49 / 48 / 46, 365 rows 28 / 28 / 28 / 28 / 30,
//   35,937 rows in 3D 66 / 66 / 60 / 60 / 60.
//   Degree 4 on 1,089 rows: 17 launched, 17 from registers, 21 through L1; degree 2 from registers costs the
//   V-cycle of that mesh 2 us.
// The coarsest level of a V-cycle is always there (at most 300 rows, or level 1).
constexpr int64_t TAIL_NNZ = 5120;
constexpr int TAIL_DEG = 5;
// Lanes per row: 4 where one thread per row would leave the chip short of loads in flight (a row
// is a chain of 21 to 100 of them), 1 from 65,536 rows on.
constexpr int64_t SPLIT_ROWS = 65536;
constexpr int TAIL_LEVELS = 24;

// sliced rows: entry j of row r at off[r / 32] + 32 j + r % 32
struct Sell {
    int64_t N = 0;
    int64_t ns = 0;            // slices
    int64_t nnz = 0;           // with padding
    int wide = 0;              // longest row; known up to TAIL_ROWS rows
    int64_t* off = nullptr;    // ns + 1
    int32_t* col = nullptr;
};

struct ChebCoef {
    float inv_theta;
    float c1[MAX_DEG], c2[MAX_DEG];
};

__device__ __forceinline__ int corner_parents(const DevMesh& m, int64_t e, int a, int p[4]) {
    const int ent = __ldg(m.e2n + e * m.nc + a);
    p[0] = ent;
    if (ent >= 0) return 1;
    const int4 hp = __ldg(reinterpret_cast<const int4*>(m.hang) - ent - 1);
    p[0] = hp.x;
    p[1] = hp.y;
    p[2] = hp.z;
    p[3] = hp.w;
    return hp.z < 0 ? 2 : 4;
}
__device__ __forceinline__ float wt_of(int n) { return n == 1 ? 1.0f : (n == 2 ? 0.5f : 0.25f); }

// ---------------- exclusive scan (int64 from int32 counts, own kernels) ----------------
constexpr int SCAN_T = 1024;
__global__ void scan_block_kernel(const int32_t* __restrict__ in, int64_t n, int64_t* __restrict__ out,
                                  int64_t* __restrict__ sums) {
    __shared__ int64_t sh[SCAN_T];
    const int64_t i = (int64_t)blockIdx.x * SCAN_T + threadIdx.x;
    const int64_t v = i < n ? in[i] : 0;
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < SCAN_T; o <<= 1) {
        const int64_t t = (int)threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    if (i < n) out[i] = sh[threadIdx.x] - v;
    if (threadIdx.x == SCAN_T - 1) sums[blockIdx.x] = sh[SCAN_T - 1];
}
// one block: sums -> exclusive prefix, total behind it
__global__ void scan_sums_kernel(int64_t* __restrict__ sums, int64_t nb) {
    __shared__ int64_t sh[SCAN_T];
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t b = 0; b < nb; b += SCAN_T) {
        const int64_t i = b + threadIdx.x;
        const int64_t v = i < nb ? sums[i] : 0;
        sh[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < SCAN_T; o <<= 1) {
            const int64_t t = (int)threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
            __syncthreads();
            sh[threadIdx.x] += t;
            __syncthreads();
        }
        if (i < nb) sums[i] = carry + sh[threadIdx.x] - v;
        __syncthreads();
        if (threadIdx.x == 0) carry += sh[SCAN_T - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[nb] = carry;
}
__global__ void scan_add_kernel(int64_t* __restrict__ out, int64_t n, const int64_t* __restrict__ sums, int64_t nb) {
    const int64_t i = (int64_t)blockIdx.x * SCAN_T + threadIdx.x;
    if (i < n) out[i] += sums[blockIdx.x];
    if (i == n) out[n] = sums[nb];
}

// ---------------- structure ----------------
// incidences of a row: (element, corner) codes e * nc + a with the row among the corner's parents
__global__ void inc_count_kernel(DevMesh m, int32_t* __restrict__ cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.E * m.nc) return;
    int p[4];
    const int n = corner_parents(m, i / m.nc, (int)(i % m.nc), p);
    for (int j = 0; j < n; ++j) atomicAdd(cnt + p[j], 1);
}
__global__ void inc_fill_kernel(DevMesh m, const int64_t* __restrict__ ip, int32_t* __restrict__ pos,
                                uint32_t* __restrict__ inc) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.E * m.nc) return;
    int p[4];
    const int n = corner_parents(m, i / m.nc, (int)(i % m.nc), p);
    for (int j = 0; j < n; ++j) inc[ip[p[j]] + atomicAdd(pos + p[j], 1)] = (uint32_t)i;
}
// ascending codes: a fixed summation order
__global__ void inc_sort_kernel(int64_t N, const int64_t* __restrict__ ip, uint32_t* __restrict__ inc) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    uint32_t* v = inc + ip[n];
    const int k = (int)(ip[n + 1] - ip[n]);
    for (int i = 1; i < k; ++i) {
        const uint32_t t = v[i];
        int j = i;
        for (; j > 0 && v[j - 1] > t; --j) v[j] = v[j - 1];
        v[j] = t;
    }
}
// Columns of a row in ascending order, one warp per row: the smallest candidate above the last
// one, until there is none (no storage, no limit on the row length).  EDGE: keep the couplings
// along an element edge.  WRITE: store them (and pad to the slice's width with the row's own
// index); otherwise the row lengths.
template <bool EDGE, bool WRITE>
__global__ void sell_cols_kernel(DevMesh m, const int64_t* __restrict__ ip, const uint32_t* __restrict__ inc,
                                 int32_t* __restrict__ rowlen, const int64_t* __restrict__ off,
                                 int32_t* __restrict__ col) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (r >= m.N) return;
    const bool skip_edge = !EDGE && m.dim == 3;
    const int64_t i0 = ip[r];
    const int n = (int)(ip[r + 1] - i0) * m.nc;
    int64_t o = 0;
    int w = 0;
    if (WRITE) {
        o = off[r >> 5];
        w = (int)((off[(r >> 5) + 1] - o) >> 5);
        o += r & 31;
    }
    int len = 0, last = -1;
    while (true) {
        int best = 0x7fffffff;
        for (int k = lane; k < n; k += 32) {
            const uint32_t code = inc[i0 + k / m.nc];
            const int b = k % m.nc;
            if (skip_edge && __popc((int)(code % m.nc) ^ b) == 1) continue;
            int p[4];
            const int np = corner_parents(m, code / m.nc, b, p);
            for (int j = 0; j < np; ++j)
                if (p[j] > last && p[j] < best) best = p[j];
        }
        best = __reduce_min_sync(0xffffffffu, best);
        if (best == 0x7fffffff) break;
        if (WRITE && lane == 0) col[o + (int64_t)len * 32] = best;
        ++len;
        last = best;
    }
    if (WRITE) {
        for (int j = len + lane; j < w; j += 32) col[o + (int64_t)j * 32] = (int32_t)r;
    } else if (lane == 0) {
        rowlen[r] = len;
    }
}
// 32 times the longest row of every slice
__global__ void sell_width_kernel(int64_t N, const int32_t* __restrict__ rowlen, int32_t* __restrict__ width) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int len = __reduce_max_sync(0xffffffffu, r < N ? rowlen[r] : 0);
    if ((threadIdx.x & 31) == 0 && r < N) width[r >> 5] = len * 32;
}
// the rows that fill up the last slice
__global__ void sell_fill_kernel(int64_t N, int64_t ns, const int64_t* __restrict__ off, int32_t* __restrict__ col) {
    const int64_t r = (ns - 1) * 32 + threadIdx.x;
    if (r < N) return;
    const int w = (int)((off[ns] - off[ns - 1]) >> 5);
    for (int j = 0; j < w; ++j) col[off[ns - 1] + (int64_t)j * 32 + threadIdx.x] = (int32_t)(N - 1);
}

// ---------------- values ----------------
struct Ref4 { float v[4]; };   // reference matrix entry by the number of axes in which two corners differ

// true length of a row: the padding repeats the row's own index, which is no larger than the
// last column, while columns ascend
__device__ __forceinline__ int row_len(const int32_t* __restrict__ c, int w) {
    int len = w;
    while (len > 1 && __ldg(c + (int64_t)(len - 1) * 32) <= __ldg(c + (int64_t)(len - 2) * 32)) --len;
    return len;
}
// Values of a row, one warp per row: the lanes form 32 element couplings (a: the row's corner,
// b: the column's corner) at a time, then every lane adds up those of the column it owns, in the
// order of the incidence list.  MASS: also the mass matrix (unit coefficients); else K with the
// element coefficients ce, without the edge couplings, its inverse diagonal and the Gershgorin
// bound of D^{-1} K.
template <bool MASS>
__global__ void sell_values_kernel(DevMesh m, Sell S, Ref4 K, Ref4 M, const int64_t* __restrict__ ip,
                                   const uint32_t* __restrict__ inc, const float* __restrict__ ce,
                                   float* __restrict__ vk, float* __restrict__ vm, float* __restrict__ dinv,
                                   unsigned int* __restrict__ kmax) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const unsigned full = 0xffffffffu;
    if (r >= S.ns * 32) return;
    const int64_t o = S.off[r >> 5] + (r & 31);
    const int w = (int)((S.off[(r >> 5) + 1] - S.off[r >> 5]) >> 5);
    if (r >= S.N) {   // fills up the last slice
        for (int j = lane; j < w; j += 32) {
            vk[o + (int64_t)j * 32] = 0.0f;
            if (MASS) vm[o + (int64_t)j * 32] = 0.0f;
        }
        return;
    }
    const int32_t* c = S.col + o;
    const int len = row_len(c, w);
    const int64_t i0 = ip[r];
    const int n = (int)(ip[r + 1] - i0) * m.nc;
    float bound = 0.0f, dg = 0.0f;
    for (int j0 = 0; j0 < w; j0 += 32) {
        const int mine = j0 + lane < len ? __ldg(c + (int64_t)(j0 + lane) * 32) : -1;
        float ak = 0.0f, am = 0.0f;
        for (int k0 = 0; k0 < n; k0 += 32) {
            const int k = k0 + lane;
            int p[4] = {-2, -2, -2, -2};
            int np = 0;
            float tk = 0.0f, tm = 0.0f;
            if (k < n) {
                const uint32_t code = inc[i0 + k / m.nc];
                const int64_t e = code / m.nc;
                const int a = (int)(code % m.nc), b = k % m.nc, diff = __popc(a ^ b);
                if (MASS || m.dim == 2 || diff != 1) {
                    np = corner_parents(m, e, a, p);
                    const float h = ldexpf((float)(m.hi - m.lo), -(int)m.level[e]);
                    const float hk = wt_of(np) * (MASS ? 1.0f : ce[e]) * (m.dim == 2 ? 1.0f : h);
                    np = corner_parents(m, e, b, p);
                    tk = hk * wt_of(np) * K.v[diff];
                    if (MASS) tm = hk * wt_of(np) * h * h * M.v[diff];
                    if (np < 2) p[1] = -2;
                    if (np < 4) p[2] = p[3] = -2;
                }
            }
            const bool hang = __any_sync(full, np > 1);
            const int cnt = min(32, n - k0);
            for (int i = 0; i < cnt; ++i) {
                const float sk = __shfl_sync(full, tk, i), sm = MASS ? __shfl_sync(full, tm, i) : 0.0f;
                bool hit = __shfl_sync(full, p[0], i) == mine;
                if (hang) {
                    const int q1 = __shfl_sync(full, p[1], i), q2 = __shfl_sync(full, p[2], i), q3 = __shfl_sync(full, p[3], i);
                    hit = hit || q1 == mine || q2 == mine || q3 == mine;   // a corner's parents differ
                }
                if (hit) {
                    ak += sk;
                    if (MASS) am += sm;
                }
            }
        }
        if (j0 + lane < w) {
            vk[o + (int64_t)(j0 + lane) * 32] = ak;
            if (MASS) vm[o + (int64_t)(j0 + lane) * 32] = am;
        }
        bound += fabsf(ak);
        if (mine == (int32_t)r) dg = ak;
    }
    if (!MASS) {
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
            bound += __shfl_xor_sync(full, bound, s);
            dg += __shfl_xor_sync(full, dg, s);
        }
        if (lane == 0) {
            const float di = dg > 0.0f ? 1.0f / dg : 0.0f, v = bound * di;
            dinv[r] = di;
            // a NaN bound reaches the check as +inf
            atomicMax(kmax, v == v ? __float_as_uint(v) : 0x7f800000u);
        }
    }
}
// A = M + eps K, its inverse diagonal and Gershgorin bound
__device__ __forceinline__ void gersh(float bound, float dinv, unsigned int* kmax) {
    float v = bound * dinv;
    const bool bad = __any_sync(0xffffffffu, !(v == v));   // fmaxf would drop a NaN
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) atomicMax(kmax, bad ? 0x7f800000u : __float_as_uint(v));
}
__global__ void sell_combine_kernel(Sell S, const float* __restrict__ vm, const float* __restrict__ vk, float eps,
                                    float* __restrict__ va, float* __restrict__ dinv, unsigned int* __restrict__ kmax) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float bound = 0.0f, di = 0.0f;
    if ((r >> 5) < S.ns) {
        const int64_t o = S.off[r >> 5] + (r & 31);
        const int w = (int)((S.off[(r >> 5) + 1] - S.off[r >> 5]) >> 5);
        float dg = 0.0f;
        for (int j = 0; j < w; ++j) {
            const int64_t s = o + (int64_t)j * 32;
            const float v = vm[s] + eps * vk[s];
            va[s] = v;
            bound += fabsf(v);
            if (S.col[s] == (int32_t)r) dg += v;   // the padding repeats the index with zeros
        }
        if (r < S.N) {
            di = dg > 0.0f ? 1.0f / dg : 0.0f;
            dinv[r] = di;
        }
    }
    gersh(bound, di, kmax);
}
// Chebyshev coefficients on [alpha, beta] (beta: 1.01 times the bound; alpha = beta / ratio, or a fixed
// alpha where ratio is 0), on the device so that no set-up waits for the host.  A block per level: the
// recurrence T_k+1 = 2 sigma T_k - T_k-1 is the serial part, one multiply-add per degree, and the quotients
// are taken by all lanes (rho_k+1 = 1 / (2 sigma - rho_k) with its two divisions: 0.6 us per degree; T_200 is
// below 1e58, as sigma <= 11/9).
struct CoefArgs {
    int deg[TAIL_LEVELS];
    double ratio[TAIL_LEVELS];
    double alpha;
};
__global__ void cheb_coef_kernel(const unsigned int* __restrict__ kmax, CoefArgs a, unsigned int bit, ChebCoef* __restrict__ out,
                                 unsigned int* __restrict__ flags) {
    const int l = blockIdx.x, deg = a.deg[l];
    const float kb = __uint_as_float(kmax[l]);
    if (!(kb > 0.0f) || isinf(kb)) {
        if (threadIdx.x == 0) atomicOr(flags, bit);
        return;
    }
    const double beta = 1.01 * (double)kb, alpha = a.ratio[l] > 0.0 ? beta / a.ratio[l] : a.alpha;
    const double theta = 0.5 * (beta + alpha), delta = 0.5 * (beta - alpha), sigma = theta / delta;
    __shared__ double T[MAX_DEG + 1];
    if (threadIdx.x == 0) {
        double t0 = 1.0, t1 = sigma;
        T[0] = t0;
        T[1] = t1;
        for (int k = 2; k <= deg; ++k) {
            const double t = fma(2.0 * sigma, t1, -t0);
            T[k] = t;
            t0 = t1;
            t1 = t;
        }
        out[l].inv_theta = (float)(1.0 / theta);
    }
    __syncthreads();
    for (int k = threadIdx.x; k + 1 < deg; k += blockDim.x) {
        out[l].c1[k] = (float)(T[k] / T[k + 2]);
        out[l].c2[k] = (float)(2.0 * T[k + 1] / (T[k + 2] * delta));
    }
}

// ---------------- row products ----------------
// row r of (val) x by LPR neighbouring lanes (all of them get the sum)
template <int LPR, class Get>
__device__ __forceinline__ float row_dot(const Sell& S, const float* __restrict__ val, int64_t r, Get x) {
    const int64_t o0 = __ldg(S.off + (r >> 5));
    const int w = (int)((__ldg(S.off + (r >> 5) + 1) - o0) >> 5), sub = LPR == 1 ? 0 : threadIdx.x % LPR;
    const float* v = val + o0 + (r & 31);
    const int32_t* c = S.col + o0 + (r & 31);
    float s = 0.0f;
#pragma unroll 8
    for (int j = sub; j < w; j += LPR) s = fmaf(__ldg(v + (int64_t)j * 32), x(__ldg(c + (int64_t)j * 32)), s);
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, LPR);
    return s;
}
// row of this thread's lane group; lanes past the end repeat the last row and store nothing
template <int LPR>
__device__ __forceinline__ int64_t my_row(int64_t N, bool& store) {
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / LPR;
    store = r < N && (LPR == 1 || threadIdx.x % LPR == 0);
    return r < N ? r : N - 1;
}

// Up to SPLIT_ROWS rows (four lanes each) the launched kernels are links of a chain: each may start
// while its predecessor runs (programmatic dependent launch), loads what no link changes (matrix,
// diagonal, coefficients), and waits there.  Every thread waits before it touches a vector, so a link
// that is done implies that all earlier ones are.  Vectors are then read with plain loads: the
// read-only path asks that nobody writes them meanwhile.  V-cycle and Cahn-Hilliard block on 45,000
// rows: 163 -> 140 us.  Larger grids fill the chip, and a successor that waits would take its place.
template <int LPR> constexpr bool LINK = LPR != 1;
template <bool ON> __device__ __forceinline__ float vec(const float* x) { return ON ? *x : __ldg(x); }
// A row of this lane group, its first PRE entries per lane already loaded
template <int LPR>
struct Row {
    static constexpr int PRE = 8;
    const float* v;
    const int32_t* c;
    int w, sub;
    float pv[PRE];
    int pc[PRE];
    __device__ __forceinline__ Row(const Sell& S, const float* __restrict__ val, int64_t r) {
        const int64_t o0 = __ldg(S.off + (r >> 5));
        w = (int)((__ldg(S.off + (r >> 5) + 1) - o0) >> 5);
        sub = threadIdx.x % LPR;
        v = val + o0 + (r & 31);
        c = S.col + o0 + (r & 31);
#pragma unroll
        for (int i = 0; i < PRE; ++i) {
            const int j = sub + i * LPR;
            pv[i] = j < w ? __ldg(v + (int64_t)j * 32) : 0.0f;
            pc[i] = j < w ? __ldg(c + (int64_t)j * 32) : (int)r;
        }
    }
    // a column scaling that no link changes
    __device__ __forceinline__ void scale(const float* __restrict__ d) {
#pragma unroll
        for (int i = 0; i < PRE; ++i) pv[i] *= __ldg(d + pc[i]);
    }
    // sum_j a_j x_j: x(column) for the loaded entries; scaled(column) brings the scaling along
    template <class X, class Scaled>
    __device__ __forceinline__ float dot(X x, Scaled scaled) const {
        float s = 0.0f;
#pragma unroll
        for (int i = 0; i < PRE; ++i) s = fmaf(pv[i], x(pc[i]), s);
#pragma unroll 8
        for (int j = sub + PRE * LPR; j < w; j += LPR) s = fmaf(__ldg(v + (int64_t)j * 32), scaled(__ldg(c + (int64_t)j * 32)), s);
#pragma unroll
        for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, LPR);
        return s;
    }
    __device__ __forceinline__ float dot(const float* x) const {
        const auto at = [&](int q) { return x[q]; };
        return dot(at, at);
    }
};
// A lane per row: nothing is loaded ahead.  The kernels are to stay at 32 registers, so that the 1,073
// blocks of 64^3 are resident at once (40 registers: 7.2 -> 9.6 us per step).
template <>
struct Row<1> {
    const Sell& S;
    const float* val;
    int64_t r;
    __device__ __forceinline__ Row(const Sell& S, const float* val, int64_t r) : S(S), val(val), r(r) {}
    __device__ __forceinline__ void scale(const float*) {}
    template <class X, class Scaled>
    __device__ __forceinline__ float dot(X, Scaled scaled) const { return row_dot<1>(S, val, r, scaled); }
    __device__ __forceinline__ float dot(const float* x) const {
        return row_dot<1>(S, val, r, [&](int q) { return __ldg(x + q); });
    }
};

// Adds m_n z_n of a block's threads to its partial; the block that finishes last sums the
// partials in a fixed order.  All threads of the block call it.
__device__ __forceinline__ void mean_add(const PrecondMean& M, double v) {
    // one warp adds up the block's values (13 FP64 instructions; a shuffle tree in every warp is 40
    // on a pipe that takes one per 16 cycles)
    __shared__ double sh[256];
    __shared__ bool last;
    const int lane = threadIdx.x;
    sh[threadIdx.x] = v;
    __syncthreads();
    if (lane < 32) {
        v = 0.0;
        for (int q = lane; q < (int)blockDim.x; q += 32) v += sh[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            M.partials[blockIdx.x] = v;
            __threadfence();
            last = atomicAdd(M.counter, 1u) == gridDim.x - 1;
            if (last) *M.counter = 0u;
        }
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    v = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) v += __ldcg(M.partials + b);
    sh[threadIdx.x] = v;
    __syncthreads();
    if (lane < 32) {
        v = 0.0;
        for (int q = lane; q < (int)blockDim.x; q += 32) v += sh[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) M.out[0] = v;
    }
}

// Chebyshev step k: r -= A d; d' = c1 d + c2 dinv r; x (+)= d.  FIRST: r is the right-hand side b
// and d = dinv b / theta is formed where it is gathered, x = 0.  LAST: the result base + x + d + d'
// goes to z (strided field f; z may be base, base may be null) and r, d' are not kept.
template <int LPR, bool FIRST, bool LAST, class TO>
__global__ void __launch_bounds__(256, LPR == 1 ? 8 : 1) cheb_step_kernel(Sell S, const float* __restrict__ val,
                                                        const float* __restrict__ dinv,
                                                        const ChebCoef* __restrict__ cf, int k, const float* b,
                                                        const float* d, float* dn, float* r, float* x, const float* base,
                                                        TO* z, int NF, int f, PrecondMean mean) {
    chain_next<LINK<LPR>>();
    bool store;
    const int64_t n = my_row<LPR>(S.N, store);
    float di, it, rr, dd, xx, y, c1, c2;
    const auto own = [&] {
        rr = FIRST ? b[n] : r[n];
        dd = FIRST ? it * di * rr : d[n];
        xx = FIRST ? 0.0f : x[n];
    };
    if constexpr (LINK<LPR>) {
        Row<LPR> row(S, val, n);
        di = dinv[n], it = FIRST ? cf->inv_theta : 0.0f, c1 = cf->c1[k], c2 = cf->c2[k];
        if (FIRST) row.scale(dinv);
        chain_wait<true>();
        own();
        y = FIRST ? it * row.dot([&](int q) { return b[q]; }, [&](int q) { return __ldg(dinv + q) * b[q]; }) : row.dot(d);
    } else {
        di = dinv[n], it = FIRST ? cf->inv_theta : 0.0f;
        own();
        if (FIRST) y = row_dot<1>(S, val, n, [&](int q) { return it * __ldg(dinv + q) * __ldg(b + q); });
        else y = row_dot<1>(S, val, n, [&](int q) { return __ldg(d + q); });
        c1 = cf->c1[k], c2 = cf->c2[k];
    }
    const float rn = rr - y, dv = c1 * dd + c2 * di * rn;
    if (LAST) {
        const float v = base ? base[n] + ((xx + dd) + dv) : (xx + dd) + dv;
        if (store) z[(size_t)n * NF + f] = (TO)v;
        if (mean.out) mean_add(mean, store ? mean.nmass[n] * (double)v : 0.0);
    } else if (store) {
        x[n] = xx + dd;
        r[n] = rn;
        dn[n] = dv;
    }
}
// t = b - A x (t may be b)
template <int LPR>
__global__ void __launch_bounds__(256, LPR == 1 ? 8 : 1) residual_kernel(Sell S, const float* __restrict__ val, const float* b, const float* x,
                                                       float* t) {
    chain_next<LINK<LPR>>();
    bool store;
    const int64_t n = my_row<LPR>(S.N, store);
    const Row<LPR> row(S, val, n);
    chain_wait<LINK<LPR>>();
    const float y = row.dot(x);
    if (store) t[n] = b[n] - y;
}
// y (+)= A x for the transfers between levels (compressed rows, 8 lanes each), a link of the chain too
template <bool ADD>
__global__ void __launch_bounds__(256) transfer_kernel(int64_t N, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                       const float* __restrict__ w, const float* x, float* y) {
    constexpr int L = 8, PRE = 4;
    chain_next<true>();
    bool store;
    const int64_t n = my_row<L>(N, store), j0 = __ldg(rp + n) + threadIdx.x % L, j1 = __ldg(rp + n + 1);
    float v[PRE], s = 0.0f;
    int c[PRE];
#pragma unroll
    for (int i = 0; i < PRE; ++i) {
        const bool has = j0 + i * L < j1;
        v[i] = has ? __ldg(w + j0 + i * L) : 0.0f;
        c[i] = has ? __ldg(col + j0 + i * L) : -1;
    }
    chain_wait<true>();
#pragma unroll
    for (int i = 0; i < PRE; ++i) s = fmaf(v[i], c[i] < 0 ? 0.0f : x[c[i]], s);
    for (int64_t j = j0 + PRE * L; j < j1; j += L) s = fmaf(__ldg(w + j), x[__ldg(col + j)], s);
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, L);
    if (store) y[n] = ADD ? y[n] + s : s;
}
// r = base + c A (x .* m): the right-hand side of a Chebyshev solve (base, m may be null)
template <int LPR>
__global__ void __launch_bounds__(256, LPR == 1 ? 8 : 1) rhs_kernel(Sell S, const float* __restrict__ val, const float* x,
                                                  const float* __restrict__ m, const float* base, float c, float* r) {
    chain_next<LINK<LPR>>();
    bool store;
    const int64_t n = my_row<LPR>(S.N, store);
    Row<LPR> row(S, val, n);
    if (m) row.scale(m);
    chain_wait<LINK<LPR>>();
    const float y = m ? row.dot([&](int q) { return vec<LINK<LPR>>(x + q); }, [&](int q) { return __ldg(m + q) * vec<LINK<LPR>>(x + q); }) : row.dot(x);
    if (store) r[n] = base ? base[n] + c * y : c * y;
}
// Cahn-Hilliard block, last pass: z_phi = x, z_mu = psi2 x + (Cn^2 K x - 2 r_mu) / m_l (lumped mass)
template <int LPR, class TO>
__global__ void __launch_bounds__(256, LPR == 1 ? 8 : 1) ch_store_kernel(Sell S, const float* __restrict__ vk, int NF, int fphi, const float* x,
                                                       const float* rm, const float* psi2, const float* __restrict__ iml,
                                                       float cn2, TO* z) {
    chain_next<LINK<LPR>>();
    bool store;
    const int64_t n = my_row<LPR>(S.N, store);
    const Row<LPR> row(S, vk, n);
    chain_wait<LINK<LPR>>();
    const float kx = row.dot(x);
    if (!store) return;
    const float xv = x[n], il = iml[n];
    z[(size_t)n * NF + fphi] = (TO)xv;
    z[(size_t)n * NF + fphi + 1] = (TO)(psi2[n] * xv + cn2 * kx * il - 2.0f * rm[n] * il);
}
// coarse element coefficients: the volume-weighted mean of the fine elements they hold
__global__ void restrict_ce_kernel(int64_t Ef, int D, const int32_t* __restrict__ fmap,
                                   const int8_t* __restrict__ lev_f, const int8_t* __restrict__ lev_c,
                                   const float* __restrict__ ce_f, float* __restrict__ ce_c) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= Ef) return;
    const int c = fmap[e];
    atomicAdd(ce_c + c, ldexpf(ce_f[e], -D * ((int)lev_f[e] - (int)lev_c[c])));
}
__global__ void iml_kernel(int64_t N, const double* __restrict__ nmass, float* __restrict__ iml) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n < N) iml[n] = 1.0f / (float)nmass[n];
}

// ---------------- small levels: one block ----------------
// Vectors that the block itself writes are read with plain loads (through L1, which is
// coherent within the block after a barrier).
struct TailLevel {
    Sell S;
    const float *val, *dinv;
    const ChebCoef* cf;
    int deg;
    float *b, *x, *t, *r, *d0, *d1;
    // transfer from this level to the next finer one (P) and its transpose
    const int64_t *rp, *rpT;
    const int32_t *col, *colT;
    const float *w, *wT;
};
struct Tail {
    int n;                 // levels, finest first
    TailLevel L[TAIL_LEVELS];
};

__device__ __forceinline__ float csr_dot(const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                                         const float* __restrict__ w, int64_t r, const float* x) {
    const int64_t j0 = __ldg(rp + r), j1 = __ldg(rp + r + 1);
    float s = 0.0f;
    for (int64_t j = j0; j < j1; ++j) s += __ldg(w + j) * x[__ldg(col + j)];
    return s;
}
// One polynomial on a level: out (+)= cheb(in); uses t, r, d0, d1.  LPR lanes per row.
template <int LPR, bool ADD>
__device__ void tail_cheb_l(const TailLevel& L, const float* in, float* out) {
    const ChebCoef* cf = L.cf;
    const float it = cf->inv_theta;
    const float* d = L.d0;
    float* dn = L.d1;
    const int64_t N = L.S.N, rounds = (N * LPR + TAIL_THREADS - 1) / TAIL_THREADS;
    const bool lead = LPR == 1 || threadIdx.x % LPR == 0;
    for (int k = 0; k + 1 < L.deg; ++k) {
        const bool last = k + 2 == L.deg;
        const float c1 = cf->c1[k], c2 = cf->c2[k];
        for (int64_t g = 0; g < rounds; ++g) {
            const int64_t q0 = (g * TAIL_THREADS + threadIdx.x) / LPR, n = q0 < N ? q0 : N - 1;
            const float di = __ldg(L.dinv + n);
            float dd, rr, xx, y;
            if (k == 0) {
                rr = in[n];
                dd = it * di * rr;
                xx = 0.0f;
                y = row_dot<LPR>(L.S, L.val, n, [&](int q) { return it * __ldg(L.dinv + q) * in[q]; });
            } else {
                rr = L.r[n];
                dd = d[n];
                xx = L.t[n];
                y = row_dot<LPR>(L.S, L.val, n, [&](int q) { return d[q]; });
            }
            const float rn = rr - y, dv = c1 * dd + c2 * di * rn;
            if (!lead || q0 >= N) continue;
            if (last) {
                const float v = (xx + dd) + dv;
                out[n] = ADD ? out[n] + v : v;
            } else {
                L.t[n] = xx + dd;
                L.r[n] = rn;
                dn[n] = dv;
            }
        }
        __syncthreads();
        const float* tmp = d;
        d = dn;
        dn = const_cast<float*>(tmp);
    }
}
// The same with everything but d in registers: a thread holds R rows of at most W entries (columns
// as 16-bit numbers), a slice of rows per warp, G entries at a time.  A step is then one gather from
// shared memory per entry and a barrier; from L1 it was three loads.
// 1,089 rows of 9 (2D), degree 16: the kernel 34 -> 18 us (and a second one of 4.6 us, which stored the
// result, went); 729 rows of 21 (3D): 17.2 -> 12.5 us; a V-cycle over 45,000 rows: 2 % of the
// application.  Half the threads with twice the rows: 17.1, 13.7 us and 2 % slower.
template <int R, int W, int G, bool ADD>
__device__ void tail_cheb_r(const TailLevel& L, const float* in, float* out, float (*sd)[TAIL_ROWS]) {
    const ChebCoef* cf = L.cf;
    const float it = __ldg(&cf->inv_theta);
    const int lane = threadIdx.x & 31, N = (int)L.S.N;
    float v[R][W], di[R], r[R], x[R], d[R];
    unsigned int c[R][W / 2];
    int w[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int s = (threadIdx.x >> 5) + i * (TAIL_THREADS / 32), n = s * 32 + lane;
        const int64_t o0 = s < L.S.ns ? __ldg(L.S.off + s) : 0;
        w[i] = s < L.S.ns ? (int)((__ldg(L.S.off + s + 1) - o0) >> 5) : 0;
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const bool has = j < w[i] && n < N;
            v[i][j] = has ? __ldg(L.val + o0 + lane + 32 * j) : 0.0f;
            const unsigned int q = has ? (unsigned int)__ldg(L.S.col + o0 + lane + 32 * j) : 0u;
            c[i][j / 2] = j & 1 ? c[i][j / 2] | q << 16 : q;
        }
        di[i] = n < N ? __ldg(L.dinv + n) : 0.0f;
        r[i] = n < N ? in[n] : 0.0f;
        d[i] = it * di[i] * r[i];
        x[i] = 0.0f;
        sd[0][n] = d[i];
    }
    float c1 = __ldg(cf->c1), c2 = __ldg(cf->c2);
    __syncthreads();
    for (int k = 0; k + 1 < L.deg; ++k) {
        const bool last = k + 2 == L.deg;
        const float* ds = sd[k & 1];
        const float n1 = last ? 0.0f : __ldg(cf->c1 + k + 1), n2 = last ? 0.0f : __ldg(cf->c2 + k + 1);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int n = (int)(threadIdx.x & ~31u) + i * TAIL_THREADS + lane;
            float y = 0.0f;
#pragma unroll
            for (int g = 0; g < W; g += G) {
                if (g >= w[i]) break;
#pragma unroll
                for (int j = g / 2; j <= (g + G - 1) / 2; ++j) asm volatile("" : "+r"(c[i][j]));   // stays packed
#pragma unroll
                for (int j = g; j < g + G; ++j)
                    y = fmaf(v[i][j], ds[j & 1 ? c[i][j / 2] >> 16 : c[i][j / 2] & 0xffffu], y);
            }
            r[i] -= y;
            x[i] += d[i];
            d[i] = c1 * d[i] + c2 * di[i] * r[i];
            if (!last) sd[(k + 1) & 1][n] = d[i];
            else if (n < N) out[n] = ADD ? out[n] + (x[i] + d[i]) : x[i] + d[i];
        }
        c1 = n1;
        c2 = n2;
        __syncthreads();
    }
}
// The register form where it fits and is long enough to pay for its loads (tail_regs tells the host); else
// from L1, eight lanes per row where that leaves one round.  (With the form handed in by the host more
// registers spill: the V-cycle of 1,049 rows takes 48 us instead of 46.)
template <bool ADD>
__device__ void tail_cheb(const TailLevel& L, const float* in, float* out, float (*sd)[TAIL_ROWS]) {
    if (L.deg >= TAIL_DEG && L.S.N <= TAIL_ROWS) {
        int w = 0;
        for (int64_t s = threadIdx.x; s < L.S.ns; s += TAIL_THREADS)
            w = max(w, (int)((__ldg(L.S.off + s + 1) - __ldg(L.S.off + s)) >> 5));
        const bool w12 = __syncthreads_and(w <= 12), w24 = __syncthreads_and(w <= 24);
        if (L.S.N <= TAIL_THREADS && w24) return tail_cheb_r<1, 24, 3, ADD>(L, in, out, sd);
        if (w12) return tail_cheb_r<2, 12, 3, ADD>(L, in, out, sd);
    }
    if (L.S.N * 8 <= TAIL_THREADS) tail_cheb_l<8, ADD>(L, in, out);
    else tail_cheb_l<1, ADD>(L, in, out);
}
// V-cycle over the block's levels (one level: its polynomial): L[0].b -> L[0].x, and to the strided
// field f of z (z not null), with its mean
template <class TO>
__global__ void __launch_bounds__(TAIL_THREADS) tail_kernel(const Tail* __restrict__ tp, TO* __restrict__ z, int NF, int f,
                                                            PrecondMean mean) {
    union Scratch { float d[2][TAIL_ROWS]; double sum[TAIL_THREADS]; };   // directions; sums of the mean
    static_assert(alignof(Scratch) >= alignof(double) && sizeof(Scratch) == sizeof(float) * 2 * TAIL_ROWS, "");
    __shared__ Scratch sm;
    float(*const sd)[TAIL_ROWS] = sm.d;
    chain_next<true>();
    chain_wait<true>();
    const Tail& T = *tp;
    const int64_t t0 = threadIdx.x, nt = TAIL_THREADS;
    for (int l = 0; l + 1 < T.n; ++l) {
        const TailLevel& L = T.L[l];
        const TailLevel& C = T.L[l + 1];
        tail_cheb<false>(L, L.b, L.x, sd);
        for (int64_t n = t0; n < L.S.N; n += nt)
            L.t[n] = L.b[n] - row_dot<1>(L.S, L.val, n, [&](int q) { return L.x[q]; });
        __syncthreads();
        for (int64_t n = t0; n < C.S.N; n += nt) C.b[n] = csr_dot(C.rpT, C.colT, C.wT, n, L.t);
        __syncthreads();
    }
    const TailLevel& B = T.L[T.n - 1];
    tail_cheb<false>(B, B.b, B.x, sd);
    for (int l = T.n - 2; l >= 0; --l) {
        const TailLevel& L = T.L[l];
        const TailLevel& C = T.L[l + 1];
        for (int64_t n = t0; n < L.S.N; n += nt) L.x[n] += csr_dot(C.rp, C.col, C.w, n, C.x);
        __syncthreads();
        for (int64_t n = t0; n < L.S.N; n += nt)
            L.b[n] -= row_dot<1>(L.S, L.val, n, [&](int q) { return L.x[q]; });
        __syncthreads();
        tail_cheb<true>(L, L.b, L.x, sd);
    }
    if (!z) return;
    const TailLevel& F = T.L[0];
    double acc = 0.0;
    for (int64_t n = t0; n < F.S.N; n += nt) {
        const float v = F.x[n];
        z[(size_t)n * NF + f] = (TO)v;
        if (mean.out) acc = fma(__ldg(mean.nmass + n), (double)v, acc);
    }
    if (!mean.out) return;
    // four warps, one per scheduler, then one
    double* const sh = sm.sum;
    sh[t0] = acc;
    __syncthreads();
    if (t0 < 128) {
        acc = 0.0;
#pragma unroll
        for (int q = 0; q < TAIL_THREADS / 128; ++q) acc += sh[t0 + 128 * q];
    }
    __syncthreads();
    if (t0 < 128) sh[t0] = acc;
    __syncthreads();
    if (t0 < 32) {
        acc = (sh[t0] + sh[t0 + 32]) + (sh[t0 + 64] + sh[t0 + 96]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (t0 == 0) mean.out[0] = acc;
    }
}
template <class T>
cudaError_t alloc(T** p, int64_t n) {
    return *p ? cudaSuccess : cudaMalloc((void**)p, (size_t)std::max<int64_t>(n, 1) * sizeof(T));
}
int blocks_for(int64_t n) { return (int)((n + 255) / 256); }

struct Level {
    DevMesh dm;
    Sell S;
    int64_t* ip = nullptr;      // incidences of every row
    uint32_t* inc = nullptr;
    float *val = nullptr, *dinv = nullptr;
    float *b = nullptr, *x = nullptr, *t = nullptr, *r = nullptr, *d0 = nullptr, *d1 = nullptr;
};

Ref4 reference(int D, bool mass) {
    // Q1 on the unit cube, 2-point Gauss (exact): products of the 1D mass (1/3, 1/6) and
    // stiffness (1, -1) entries; by symmetry only the number of differing axes matters
    Ref4 R{};
    for (int d = 0; d <= D; ++d) {
        auto m1 = [&](int k) { return k < d ? 1.0 / 6.0 : 1.0 / 3.0; };   // axis k differs when k < d
        double s = 0.0;
        if (mass) {
            s = 1.0;
            for (int k = 0; k < D; ++k) s *= m1(k);
        } else {
            for (int k = 0; k < D; ++k) {
                double p = k < d ? -1.0 : 1.0;
                for (int j = 0; j < D; ++j)
                    if (j != k) p *= m1(j);
                s += p;
            }
        }
        R.v[d] = (float)s;
    }
    return R;
}

}  // namespace

struct PrecondWS {
    std::vector<Level> lv;       // 0: the mesh; more once a V-cycle was asked for
    ChebCoef* cf = nullptr;      // TAIL_LEVELS of the Schur levels, one of the Cahn-Hilliard block
    unsigned int* kmax = nullptr;
    unsigned int* flags = nullptr;
    // Cahn-Hilliard block on the mesh
    Sell SC;
    float *vm = nullptr, *vk = nullptr, *va = nullptr, *ch_dinv = nullptr, *iml = nullptr, *rm = nullptr, *rp = nullptr,
          *cb = nullptr, *ca = nullptr, *cr = nullptr, *cx = nullptr, *cd0 = nullptr, *cd1 = nullptr;
    const float* psi2 = nullptr;
    Tail* tail = nullptr;        // device descriptor of the one-block kernel's levels
    int tail_from = -1, tail_deg = 0;
    bool tail_mg = false;
    cudaStream_t cap = nullptr, cap2 = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    bool no_graphs = false;
    struct Graph {
        cudaGraphExec_t exec = nullptr;
        const void *mean = nullptr, *z = nullptr;
        size_t to = 0;
        PrecondSpec spec;
        int nk = 0;
    } graph[4];
    int next = 0;
};

namespace {

// exclusive scan of n counts into out[0..n]; total to *total (synchronises)
cudaError_t scan(const int32_t* in, int64_t n, int64_t* out, int64_t* total, cudaStream_t s) {
    const int64_t nb = (n + SCAN_T - 1) / SCAN_T;
    int64_t* sums = nullptr;
    cudaError_t e = cudaMalloc((void**)&sums, (size_t)(nb + 1) * sizeof(int64_t));
    if (e != cudaSuccess) return e;
    scan_block_kernel<<<(unsigned)nb, SCAN_T, 0, s>>>(in, n, out, sums);
    scan_sums_kernel<<<1, SCAN_T, 0, s>>>(sums, nb);
    scan_add_kernel<<<(unsigned)(n / SCAN_T + 1), SCAN_T, 0, s>>>(out, n, sums, nb);
    chns_count_launches(3);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(total, sums + nb, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(sums);
    return e;
}
void sell_free(Sell& S) {
    cudaFree(S.off);
    cudaFree(S.col);
    S = Sell();
}
// incidences (once per level) and the column structure
cudaError_t inc_build(Level& L, cudaStream_t s) {
    if (L.ip) return cudaSuccess;
    const DevMesh& m = L.dm;
    int32_t* cnt = nullptr;
    int64_t total = 0;
    cudaError_t e = alloc(&cnt, m.N);
    if (e == cudaSuccess) e = alloc(&L.ip, m.N + 1);
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (size_t)m.N * sizeof(int32_t), s);
    if (e == cudaSuccess) {
        inc_count_kernel<<<blocks_for(m.E * m.nc), 256, 0, s>>>(m, cnt);
        chns_count_launches(1);
        e = scan(cnt, m.N, L.ip, &total, s);
    }
    if (e == cudaSuccess) e = alloc(&L.inc, total);
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, (size_t)m.N * sizeof(int32_t), s);
    if (e == cudaSuccess) {
        inc_fill_kernel<<<blocks_for(m.E * m.nc), 256, 0, s>>>(m, L.ip, cnt, L.inc);
        inc_sort_kernel<<<blocks_for(m.N), 256, 0, s>>>(m.N, L.ip, L.inc);
        chns_count_launches(2);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(cnt);
    if (e != cudaSuccess) {
        cudaFree(L.ip);
        cudaFree(L.inc);
        L.ip = nullptr;
        L.inc = nullptr;
    }
    return e;
}
template <bool EDGE>
cudaError_t sell_build(const Level& L, Sell& S, cudaStream_t s) {
    if (S.col) return cudaSuccess;
    const DevMesh& m = L.dm;
    Sell T;
    T.N = m.N;
    T.ns = (m.N + 31) / 32;
    int32_t *width = nullptr, *len = nullptr;
    cudaError_t e = alloc(&width, T.ns);
    if (e == cudaSuccess) e = alloc(&len, m.N);
    if (e == cudaSuccess) e = alloc(&T.off, T.ns + 1);
    if (e == cudaSuccess) {
        sell_cols_kernel<EDGE, false><<<blocks_for(m.N * 32), 256, 0, s>>>(m, L.ip, L.inc, len, nullptr, nullptr);
        sell_width_kernel<<<blocks_for(m.N), 256, 0, s>>>(m.N, len, width);
        chns_count_launches(2);
        e = scan(width, T.ns, T.off, &T.nnz, s);
    }
    if (e == cudaSuccess && m.N <= TAIL_ROWS) {
        int32_t w[TAIL_ROWS / 32];
        e = cudaMemcpyAsync(w, width, (size_t)T.ns * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e == cudaSuccess) T.wide = *std::max_element(w, w + T.ns) / 32;
    }
    if (e == cudaSuccess) e = alloc(&T.col, T.nnz);
    if (e == cudaSuccess) {
        sell_cols_kernel<EDGE, true><<<blocks_for(m.N * 32), 256, 0, s>>>(m, L.ip, L.inc, nullptr, T.off, T.col);
        sell_fill_kernel<<<1, 32, 0, s>>>(m.N, T.ns, T.off, T.col);
        chns_count_launches(2);
        e = cudaGetLastError();
    }
    cudaFree(len);
    cudaFree(width);
    if (e != cudaSuccess) sell_free(T);
    else S = T;
    return e;
}
cudaError_t level_alloc(Level& L, cudaStream_t s) {
    cudaError_t e = inc_build(L, s);
    if (e == cudaSuccess) e = sell_build<false>(L, L.S, s);
    if (e == cudaSuccess) e = alloc(&L.val, L.S.nnz);
    for (float** p : {&L.dinv, &L.b, &L.x, &L.t, &L.r, &L.d0, &L.d1})
        if (e == cudaSuccess) e = alloc(p, L.dm.N);
    return e;
}
void level_free(Level& L) {
    sell_free(L.S);
    cudaFree(L.ip);
    cudaFree(L.inc);
    for (float* p : {L.val, L.dinv, L.b, L.x, L.t, L.r, L.d0, L.d1}) cudaFree(p);
}
int level_degree(const PrecondWS* p, const PrecondSpec& spec, int l) {
    return spec.mg && l + 1 == (int)p->lv.size() ? COARSE_DEG : spec.degree;
}
// whether tail_cheb takes the register form for a level
bool tail_regs(const Sell& S, int deg) {
    return deg >= TAIL_DEG && ((S.N <= TAIL_THREADS && S.wide <= 24) || (S.N <= TAIL_ROWS && S.wide <= 12));
}
// first level of the one-block kernel: 0 when the whole operator runs there, the number of levels when a
// polynomial does not use it (a V-cycle always does)
int first_tail(const PrecondWS* p, const PrecondSpec& spec) {
    const int nl = spec.mg ? (int)p->lv.size() : 1;
    for (int l = 0; l < nl; ++l) {
        const Sell& S = p->lv[(size_t)l].S;
        if (S.nnz <= TAIL_NNZ || tail_regs(S, level_degree(p, spec, l))) return l;
    }
    return spec.mg ? nl - 1 : nl;
}
chns_status tail_describe(chns_mesh* m, const PrecondSpec& spec) {
    PrecondWS* p = m->pre;
    const int from = first_tail(p, spec), nl = spec.mg ? (int)p->lv.size() : 1;
    if (p->tail && p->tail_from == from && p->tail_deg == spec.degree && p->tail_mg == spec.mg) return CHNS_OK;
    precond_drop_graphs(m);   // they hold the old description
    if (!p->tail) CHNS_CUDA(cudaMalloc((void**)&p->tail, sizeof(Tail)));
    std::vector<unsigned char> raw(sizeof(Tail), 0);
    Tail& T = *reinterpret_cast<Tail*>(raw.data());
    T.n = std::max(nl - from, 0);
    for (int l = from; l < nl; ++l) {
        const Level& L = p->lv[(size_t)l];
        TailLevel& t = T.L[l - from];
        t.S = L.S;
        t.val = L.val;
        t.dinv = L.dinv;
        t.cf = p->cf + l;
        t.deg = level_degree(p, spec, l);
        t.b = L.b;
        t.x = L.x;
        t.t = L.t;
        t.r = L.r;
        t.d0 = L.d0;
        t.d1 = L.d1;
        if (l > 0) {
            const TransferDev& P = m->mg->lv[(size_t)l].P;
            t.rp = P.rp;
            t.col = P.col;
            t.w = P.wf;
            t.rpT = P.rpT;
            t.colT = P.colT;
            t.wT = P.wTf;
        }
    }
    CHNS_CUDA(cudaMemcpy(p->tail, &T, sizeof(Tail), cudaMemcpyHostToDevice));
    p->tail_from = from;
    p->tail_deg = spec.degree;
    p->tail_mg = spec.mg;
    return CHNS_OK;
}

// f with the lanes per row for N rows
template <class F>
void split(int64_t N, F f) {
    if (N < SPLIT_ROWS) f(std::integral_constant<int, 4>());
    else f(std::integral_constant<int, 1>());
}
void launch_residual_rows(const Level& L, float* t, cudaStream_t st) {   // t = b - A x
    split(L.dm.N, [&](auto lpr) {
        constexpr int LPR = decltype(lpr)::value;
        chain<LINK<LPR>>(residual_kernel<LPR>, blocks_for(L.dm.N * LPR), 256, st, L.S, L.val, L.b, L.x, t);
    });
}

// z = base + polynomial of b (b is not x); the pressure's mean with it where asked for
template <class TO>
int cheb(const Sell& S, const float* val, const float* dinv, const ChebCoef* cf, int deg, const float* b, float* r, float* x,
         float* d0, float* d1, const float* base, TO* z, int NF, int f, const PrecondMean& mean, cudaStream_t st) {
    split(S.N, [&](auto lpr) {
        constexpr int LPR = decltype(lpr)::value;
        const int g = blocks_for(S.N * LPR);
        for (int k = 0; k + 1 < deg; ++k) {
            const bool last = k + 2 == deg;
            auto run = [&](auto first, auto fin) {
                chain<LINK<LPR>>(cheb_step_kernel<LPR, decltype(first)::value, decltype(fin)::value, TO>, g, 256, st, S, val, dinv, cf, k, b, d0,
                      d1, r, x, base, z, NF, f, mean);
            };
            if (k == 0 && last) run(std::true_type(), std::true_type());
            else if (k == 0) run(std::true_type(), std::false_type());
            else if (last) run(std::false_type(), std::true_type());
            else run(std::false_type(), std::false_type());
            std::swap(d0, d1);
        }
    });
    return deg - 1;
}
// z = base + polynomial of the level's b
template <class TO>
int smooth(const Level& L, const ChebCoef* cf, int deg, const float* base, TO* z, int NF, int f, const PrecondMean& mean,
           cudaStream_t st) {
    return cheb<TO>(L.S, L.val, L.dinv, cf, deg, L.b, L.r, L.t, L.d0, L.d1, base, z, NF, f, mean, st);
}
// One V-cycle from level 0's b, result to field f of z: on every level pre-smoothing from 0,
// residual, restriction, the coarser cycle, prolongation, residual (in place of b), post-smoothing.
template <class TO>
cudaError_t vcycle(chns_mesh* m, const PrecondSpec& spec, TO* z, int NF, int f, const PrecondMean& mean, cudaStream_t st,
                   int* nk) {
    PrecondWS* p = m->pre;
    const int from = p->tail_from;
    for (int l = 0; l < from; ++l) {
        Level& L = p->lv[(size_t)l];
        *nk += smooth<float>(L, p->cf + l, spec.degree, nullptr, L.x, 1, 0, PrecondMean(), st);
        launch_residual_rows(L, L.t, st);
        const TransferDev& P = m->mg->lv[(size_t)l + 1].P;
        chain<true>(transfer_kernel<false>, blocks_for(P.n_src * 8), 256, st, P.n_src, P.rpT, P.colT, P.wTf, L.t, p->lv[(size_t)l + 1].b);
        *nk += 2;
    }
    const bool all = from == 0;   // every level runs in the one block
    chain<true>(tail_kernel<TO>, 1, TAIL_THREADS, st, p->tail, all ? z : nullptr, NF, f, all ? mean : PrecondMean());
    ++*nk;
    for (int l = from - 1; l >= 0; --l) {
        Level& L = p->lv[(size_t)l];
        const TransferDev& P = m->mg->lv[(size_t)l + 1].P;
        chain<true>(transfer_kernel<true>, blocks_for(P.n_dst * 8), 256, st, P.n_dst, P.rp, P.col, P.wf, p->lv[(size_t)l + 1].x, L.x);
        launch_residual_rows(L, L.b, st);
        *nk += 2;
        *nk += l == 0 ? smooth<TO>(L, p->cf, spec.degree, L.x, z, NF, f, mean, st)
                      : smooth<float>(L, p->cf + l, spec.degree, L.x, L.x, 1, 0, PrecondMean(), st);
    }
    return cudaGetLastError();
}
template <class TO>
cudaError_t polynomial(chns_mesh* m, const PrecondSpec& spec, TO* z, int NF, int f, const PrecondMean& mean, cudaStream_t st,
                       int* nk) {
    PrecondWS* p = m->pre;
    Level& L = p->lv[0];
    if (p->tail_from == 0) {
        chain<true>(tail_kernel<TO>, 1, TAIL_THREADS, st, p->tail, z, NF, f, mean);
        ++*nk;
        return cudaGetLastError();
    }
    *nk += smooth<TO>(L, p->cf, spec.degree, nullptr, z, NF, f, mean, st);
    return cudaGetLastError();
}
// phi and mu: mu eliminated with the lumped mass, the phi Schur complement by two polynomials
template <class TO>
cudaError_t cahn_hilliard(chns_mesh* m, const PrecondSpec& spec, TO* z, int NF, int f, cudaStream_t st, int* nk) {
    PrecondWS* p = m->pre;
    const int64_t N = m->dm.N;
    const ChebCoef* cf = p->cf + TAIL_LEVELS;
    auto rhs = [&](const float* val, const float* x, const float* mul, const float* base, float a, float* r) {
        split(N, [&](auto lpr) {
            constexpr int LPR = decltype(lpr)::value;
            chain<LINK<LPR>>(rhs_kernel<LPR>, blocks_for(N * LPR), 256, st, p->SC, val, x, mul, base, a, r);
        });
    };
    auto solve = [&](const float* b, float* x) {   // (M + eps K)^{-1} b
        return cheb<float>(p->SC, p->va, p->ch_dinv, cf, CH_DEG, b, p->cr, p->cx, p->cd0, p->cd1, nullptr, x, 1, 0, PrecondMean(), st);
    };
    rhs(p->vk, p->rm, p->iml, p->rp, spec.inv_pecn, p->cb);   // r_phi + K M_L^{-1} r_mu / (Pe Cn)
    *nk += 1 + solve(p->cb, p->ca);
    rhs(p->vm, p->ca, nullptr, nullptr, spec.dt, p->cb);      // dt M s
    *nk += 2 + solve(p->cb, p->ca);
    split(N, [&](auto lpr) {
        constexpr int LPR = decltype(lpr)::value;
        chain<LINK<LPR>>(ch_store_kernel<LPR, TO>, blocks_for(N * LPR), 256, st, p->SC, p->vk, NF, f, p->ca, p->rm, p->psi2, p->iml, spec.cn2, z);
    });
    return cudaGetLastError();
}
template <class TO>
cudaError_t enqueue(chns_mesh* m, const PrecondSpec& spec, TO* z, const PrecondMean& mean, cudaStream_t st, cudaStream_t side,
                    int* nk) {
    PrecondWS* p = m->pre;
    const int D = m->dm.dim, NF = m->dm.nf;
    cudaError_t e = cudaSuccess;
    // the pressure and the Cahn-Hilliard chains are independent: two branches of the graph
    const bool both = spec.schur && spec.ch && side;
    if (both) {
        e = cudaEventRecord(p->fork, st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(side, p->fork, 0);
        if (e != cudaSuccess) return e;
    }
    if (spec.ch) e = cahn_hilliard<TO>(m, spec, z, NF, D + 1, both ? side : st, nk);
    if (e == cudaSuccess && spec.schur)
        e = spec.mg ? vcycle<TO>(m, spec, z, NF, D, mean, st, nk) : polynomial<TO>(m, spec, z, NF, D, mean, st, nk);
    if (both) {
        const cudaError_t e1 = cudaEventRecord(p->join, side);
        const cudaError_t e2 = cudaStreamWaitEvent(st, p->join, 0);
        if (e == cudaSuccess) e = e1 != cudaSuccess ? e1 : e2;
    }
    return e;
}

template <class TO>
chns_status apply_any(chns_mesh* m, const PrecondSpec& spec, TO* z, const PrecondMean& mean, cudaStream_t s) {
    PrecondWS* p = m->pre;
    if (!p->no_graphs) {
        PrecondWS::Graph* hit = nullptr;
        for (auto& g : p->graph)
            if (g.exec && g.z == (const void*)z && g.to == sizeof(TO) && g.mean == (const void*)mean.out && g.spec == spec) hit = &g;
        if (!hit) {
            PrecondWS::Graph* slot = &p->graph[p->next];
            cudaGraph_t gr = nullptr;
            cudaGraphExec_t ex = nullptr;
            int nk = 0;
            bool ok = cudaStreamBeginCapture(p->cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
            if (ok) {
                ok = enqueue<TO>(m, spec, z, mean, p->cap, p->cap2, &nk) == cudaSuccess;
                ok = (cudaStreamEndCapture(p->cap, &gr) == cudaSuccess) && ok && gr != nullptr;
                if (ok) ok = cudaGraphInstantiate(&ex, gr, 0) == cudaSuccess;
                if (gr) cudaGraphDestroy(gr);
            }
            if (!ok) {
                (void)cudaGetLastError();   // capture unavailable: launch directly from now on
                p->no_graphs = true;
            } else {
                if (slot->exec) cudaGraphExecDestroy(slot->exec);
                slot->exec = ex;
                slot->mean = mean.out;
                slot->z = z;
                slot->to = sizeof(TO);
                slot->spec = spec;
                slot->nk = nk;
                p->next = (p->next + 1) % 4;
                hit = slot;
            }
        }
        if (hit) {
            CHNS_CUDA(cudaGraphLaunch(hit->exec, s));
            chns_count_launches(hit->nk);
            return CHNS_OK;
        }
    }
    int nk = 0;
    CHNS_CUDA(enqueue<TO>(m, spec, z, mean, s, nullptr, &nk));
    chns_count_launches(nk);
    return CHNS_OK;
}

}  // namespace

chns_status precond_prepare(chns_mesh* m, const PrecondSpec& spec, cudaStream_t s) {
    if (!m->pre) {
        m->pre = new (std::nothrow) PrecondWS();
        if (!m->pre) { chns_set_error("host allocation failed"); return CHNS_ENOMEM; }
    }
    PrecondWS* p = m->pre;
    if (!p->cap) {
        CHNS_CUDA(cudaStreamCreateWithFlags(&p->cap, cudaStreamNonBlocking));
        CHNS_CUDA(cudaStreamCreateWithFlags(&p->cap2, cudaStreamNonBlocking));
        CHNS_CUDA(cudaEventCreateWithFlags(&p->fork, cudaEventDisableTiming));
        CHNS_CUDA(cudaEventCreateWithFlags(&p->join, cudaEventDisableTiming));
    }
    CHNS_CUDA(alloc(&p->cf, TAIL_LEVELS + 1));
    CHNS_CUDA(alloc(&p->kmax, TAIL_LEVELS + 1));
    CHNS_CUDA(alloc(&p->flags, 1));
    if (p->lv.empty()) {
        p->lv.emplace_back();
        p->lv[0].dm = m->dm;
    }
    if (spec.schur) {
        if (spec.mg) {
            chns_status st = mg_hier_build(m);
            if (st != CHNS_OK) return st;
            for (size_t l = p->lv.size(); l < m->mg->lv.size(); ++l) {
                p->lv.emplace_back();
                p->lv[l].dm = m->mg->lv[l].dm;
            }
        }
        for (size_t l = 0; l < (spec.mg ? p->lv.size() : 1); ++l)
            if (!p->lv[l].d1) CHNS_CUDA(level_alloc(p->lv[l], s));
        chns_status st = tail_describe(m, spec);
        if (st != CHNS_OK) return st;
    }
    if (spec.ch && !p->cd1) {
        Level& L = p->lv[0];
        const int64_t N = m->dm.N;
        CHNS_CUDA(inc_build(L, s));
        CHNS_CUDA(sell_build<true>(L, p->SC, s));
        for (float** a : {&p->vm, &p->vk, &p->va}) CHNS_CUDA(alloc(a, p->SC.nnz));
        for (float** a : {&p->ch_dinv, &p->iml, &p->rm, &p->rp, &p->cb, &p->ca, &p->cr, &p->cx, &p->cd0}) CHNS_CUDA(alloc(a, N));
        iml_kernel<<<blocks_for(N), 256, 0, s>>>(N, m->d_nmass, p->iml);
        sell_values_kernel<true><<<blocks_for(p->SC.ns * 1024), 256, 0, s>>>(m->dm, p->SC, reference(m->dm.dim, false),
                                                                             reference(m->dm.dim, true), L.ip, L.inc, nullptr,
                                                                             p->vk, p->vm, nullptr, nullptr);
        chns_count_launches(2);
        CHNS_CUDA(cudaGetLastError());
        CHNS_CUDA(alloc(&p->cd1, N));
    }
    return CHNS_OK;
}

chns_status precond_setup(chns_mesh* m, const PrecondSpec& spec, const float* ce, const float* psi2, cudaStream_t s) {
    PrecondWS* p = m->pre;
    CHNS_CUDA(cudaMemsetAsync(p->flags, 0, sizeof(unsigned int), s));
    CHNS_CUDA(cudaMemsetAsync(p->kmax, 0, (TAIL_LEVELS + 1) * sizeof(unsigned int), s));
    if (spec.schur) {
        const Ref4 K = reference(m->dm.dim, false);
        const int nl = spec.mg ? (int)p->lv.size() : 1;
        CoefArgs ca = {};
        for (int l = 0; l < nl; ++l) {
            Level& L = p->lv[(size_t)l];
            const float* cel = ce;
            if (l > 0) {
                MGLevel& C = m->mg->lv[(size_t)l];
                MGLevel& F = m->mg->lv[(size_t)l - 1];
                CHNS_CUDA(cudaMemsetAsync(C.ce, 0, (size_t)C.E * sizeof(float), s));
                restrict_ce_kernel<<<blocks_for(F.E), 256, 0, s>>>(F.E, m->dm.dim, C.fmap, F.dm.level, C.dm.level,
                                                                   l == 1 ? ce : F.ce, C.ce);
                chns_count_launches(1);
                cel = C.ce;
            }
            sell_values_kernel<false><<<blocks_for(L.S.ns * 1024), 256, 0, s>>>(L.dm, L.S, K, K, L.ip, L.inc, cel, L.val, nullptr,
                                                                                L.dinv, p->kmax + l);
            chns_count_launches(1);
            ca.deg[l] = level_degree(p, spec, l);
            // smoother: the upper part of the spectrum of D^{-1} K; polynomial and coarsest level: all of it
            const double nside = std::ldexp(1.0, l == 0 ? m->max_level : m->mg->lv[(size_t)l].mesh->max_level);
            ca.ratio[l] = spec.mg && l + 1 < nl ? 10.0 : std::max(16.0, nside * nside / 8.0);
        }
        cheb_coef_kernel<<<nl, 128, 0, s>>>(p->kmax, ca, 1u, p->cf, p->flags);
        chns_count_launches(1);
    }
    if (spec.ch) {
        if (p->psi2 != psi2) {
            precond_drop_graphs(m);
            p->psi2 = psi2;
        }
        sell_combine_kernel<<<blocks_for(m->dm.N), 256, 0, s>>>(p->SC, p->vm, p->vk, spec.eps, p->va, p->ch_dinv,
                                                                p->kmax + TAIL_LEVELS);
        CoefArgs ca = {};
        ca.deg[0] = CH_DEG;
        ca.alpha = 0.05;
        cheb_coef_kernel<<<1, 32, 0, s>>>(p->kmax + TAIL_LEVELS, ca, 2u, p->cf + TAIL_LEVELS, p->flags);
        chns_count_launches(2);
    }
    CHNS_CUDA(cudaGetLastError());
    return CHNS_OK;
}

const unsigned int* precond_flags(const chns_mesh* m) { return m->pre->flags; }

chns_status precond_apply(chns_mesh* m, const PrecondSpec& spec, float* z, const PrecondMean& mean, cudaStream_t s) {
    return apply_any(m, spec, z, mean, s);
}
chns_status precond_apply(chns_mesh* m, const PrecondSpec& spec, double* z, const PrecondMean& mean, cudaStream_t s) {
    return apply_any(m, spec, z, mean, s);
}
PrecondIn precond_inputs(const chns_mesh* m) {
    PrecondIn in;
    if (!m->pre->lv.empty()) in.p = m->pre->lv[0].b;
    in.phi = m->pre->rp;
    in.mu = m->pre->rm;
    return in;
}

void precond_drop_graphs(chns_mesh* m) {
    if (!m->pre) return;
    for (auto& g : m->pre->graph) {
        if (g.exec) cudaGraphExecDestroy(g.exec);
        g = PrecondWS::Graph();
    }
}

void precond_free(PrecondWS* p) {
    if (!p) return;
    for (auto& g : p->graph)
        if (g.exec) cudaGraphExecDestroy(g.exec);
    for (auto& L : p->lv) level_free(L);
    sell_free(p->SC);
    for (float* a : {p->vm, p->vk, p->va, p->ch_dinv, p->iml, p->rm, p->rp, p->cb, p->ca, p->cr, p->cx, p->cd0, p->cd1}) cudaFree(a);
    cudaFree(p->cf);
    cudaFree(p->kmax);
    cudaFree(p->flags);
    cudaFree(p->tail);
    if (p->fork) cudaEventDestroy(p->fork);
    if (p->join) cudaEventDestroy(p->join);
    if (p->cap) cudaStreamDestroy(p->cap);
    if (p->cap2) cudaStreamDestroy(p->cap2);
    delete p;
}
