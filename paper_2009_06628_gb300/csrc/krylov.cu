// Vector kernels of the Arnoldi process (Newton's GMRES and the adjoint's), FP64.
//
// The basis is kept unnormalised: slot j of V holds w_j and a device scalar s_j = 1/|w_j|, and
// v_j = s_j w_j.  The scale rides along where a vector is read anyway, so no pass normalises.
// One Gram-Schmidt pass is a dot kernel (forming w = S y + mean on the way) and an update kernel with
// the new norm; the last block of each sums the partials, in a fixed order, and the update's writes
// what the host waits for into pinned memory.  A second pass is queued behind the first and decided on
// the device: its blocks return at once when |w| kept a tenth of its length.  (Left to the host, it
// costs a discarded operator application whenever it is wanted, which is often: two drops, 81 -> 118 ms
// per Newton step.)
//
// Bound: k FP64 FMAs per entry and pass on the narrow FP64 pipe (n = 1.65 M, k = 15: 39 us) next
// to one read of V (29 us).  Three splits of that work, by size (orthogonalise):
// long vectors: one kernel per number of columns (dots) or per remainder (update), so that all loads
// of an entry pair go out together, and few threads take many rows, so that the reductions add 5 % of
// FP64 work.  The update walks the rows backwards, where the dot pass has just left its columns in L2
// (evict-first loads there: 34 -> 50 us).
//   n = 1.65 M, k = 1..30: dots 3.3 us per column + 24 us (w formed, 4 us of reduction), update
//   2.7 us per column + 10 us; all of an Arnoldi step's vector work 181 -> 136 us, and without the
//   33 us of the normalising, scaling and mean passes that it takes in.
// shorter ones: the columns go over the grid too, 8 per block, and several lanes share the columns of a
// pair in the update; the shortest, with few columns: one cluster of 16 blocks.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "chns_internal.h"
#include "krylov.h"

namespace krylov {

namespace {

__device__ __forceinline__ double formed(const Source& s, int64_t i, double mean) {
    const double y = s.yf ? (double)s.yf[i] : s.yd[i];
    const double w = s.S[i] * y;
    return s.mean && (int)((uint32_t)i % (uint32_t)s.NF) == s.f ? w + mean : w;   // n < 2^32
}

// sums of KP numbers (a power of two, at most 32) over the warp: halved over the lanes, then one
// number per lane group.  Sum number `returned` ends up in acc[0].
template <int KP>
__device__ __forceinline__ int warp_sums(double* acc, int lane) {
    int base = 0, cnt = KP;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        if (cnt > 1) {
            cnt /= 2;
            const bool up = lane & o;
#pragma unroll
            for (int t = 0; t < KP / 2; ++t) {
                if (t >= cnt) break;
                const double keep = up ? acc[cnt + t] : acc[t], give = up ? acc[t] : acc[cnt + t];
                acc[t] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
            base += up ? cnt : 0;
        } else {
            acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
        }
    }
    return base;
}

// h = s .* (V^T w) for K <= 32 columns starting at V, and |w|^2 (nrm not null).  With a source w is
// formed here and slot w gets it.  pred: return unless it is 1.
template <int K>
__global__ void __launch_bounds__(T, 2)
dots_kernel(const double* __restrict__ V, int64_t ld, Source src, double* w, int64_t n, const double* __restrict__ scale,
            double* __restrict__ h, double* __restrict__ nrm, double* __restrict__ partials, unsigned int* counter,
            const double* __restrict__ pred) {
    if (pred && pred[0] == 0.0) return;
    constexpr int KP = K <= 1 ? 1 : K <= 2 ? 2 : K <= 4 ? 4 : K <= 8 ? 8 : K <= 16 ? 16 : 32;   // halves evenly
    double acc[KP], nn = 0.0;
#pragma unroll
    for (int j = 0; j < KP; ++j) acc[j] = 0.0;
    const bool form = src.yf || src.yd;
    const double mean = src.mean ? src.a * src.mean[0] : 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * 2, full_pairs = n / 2 * 2;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 2; i < full_pairs; i += stride) {
        double2 x;
        if (form) {
            x = make_double2(formed(src, i, mean), formed(src, i + 1, mean));
            *reinterpret_cast<double2*>(w + i) = x;
        } else {
            x = *reinterpret_cast<const double2*>(w + i);
        }
        const double* p = V + i;
        // the columns' loads are independent: as many in flight as the registers hold
        double2 v[K];
#pragma unroll
        for (int j = 0; j < K; ++j) v[j] = *reinterpret_cast<const double2*>(p + (size_t)j * ld);
        if (nrm) nn = fma(x.y, x.y, fma(x.x, x.x, nn));
#pragma unroll
        for (int j = 0; j < K; ++j) acc[j] = fma(v[j].y, x.y, fma(v[j].x, x.x, acc[j]));
    }
    if (full_pairs < n && blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t i = n - 1;
        const double x = form ? formed(src, i, mean) : w[i];
        if (form) w[i] = x;
        nn = fma(x, x, nn);
#pragma unroll
        for (int j = 0; j < K; ++j) acc[j] = fma(V[(size_t)j * ld + i], x, acc[j]);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, base = warp_sums<KP>(acc, lane);
    __shared__ double sh[T / 32][KP + 1];
    __shared__ double fin[T];
    sh[warp][base] = acc[0];   // lanes that share a number hold the same sum
    if (nrm) {
        nn = warp_sum(nn);
        if (lane == 0) sh[warp][KP] = nn;
    }
    __syncthreads();
    if (threadIdx.x <= KP && (threadIdx.x < KP || nrm)) {
        double v = 0.0;
        for (int q = 0; q < (int)blockDim.x / 32; ++q) v += sh[q][threadIdx.x];
        partials[(size_t)blockIdx.x * (KP + 1) + threadIdx.x] = v;
    }
    if (!last_block(counter)) return;
    // thread (g, j) adds up number j of blocks g, g + groups, ...: eight loads in flight, so that this
    // tail is a few memory latencies long
    const int groups = blockDim.x / KP, g = threadIdx.x / KP, num = threadIdx.x % KP;
    double v = 0.0;
#pragma unroll 8
    for (int b = g; b < (int)gridDim.x; b += groups) v += __ldcg(partials + (size_t)b * (KP + 1) + num);
    fin[threadIdx.x] = v;
    if (nrm) {
        double t = 0.0;
#pragma unroll 4
        for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) t += __ldcg(partials + (size_t)b * (KP + 1) + KP);
        t = warp_sum(t);
        if (lane == 0) sh[warp][KP] = t;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double t = 0.0;
#pragma unroll 8
        for (int q = 0; q < groups; ++q) t += fin[q * KP + threadIdx.x];
        h[threadIdx.x] = t * scale[threadIdx.x];
    }
    if (nrm && threadIdx.x == blockDim.x - 1) {
        double t = 0.0;
        for (int q = 0; q < (int)blockDim.x / 32; ++q) t += sh[q][KP];
        nrm[0] = t;
    }
}

// The same for all k columns in one launch, C of them per row of the grid: vectors too short for the
// kernel above to fill the chip with rows alone, which also takes 32 columns per launch.  Every chunk
// forms w for itself, the first stores it.  Columns past the last repeat it and are dropped.  counter:
// one per chunk.
template <int C>
__global__ void __launch_bounds__(T, 2)
dots_chunks_kernel(const double* __restrict__ V, int64_t ld, int k, Source src, double* w, int64_t n, const double* __restrict__ scale,
                   double* __restrict__ h, double* __restrict__ nrm, double* __restrict__ partials, unsigned int* counter,
                   const double* __restrict__ pred) {
    if (pred && pred[0] == 0.0) return;
    const int j0 = blockIdx.y * C;
    const bool first = blockIdx.y == 0, form = src.yf || src.yd;
    const double mean = src.mean ? src.a * src.mean[0] : 0.0;
    const double* col[C];
    double acc[C], nn = 0.0;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        col[j] = V + (size_t)min(j0 + j, k - 1) * ld;
        acc[j] = 0.0;
    }
    const int64_t stride = (int64_t)gridDim.x * T * 2;
    for (int64_t i = ((int64_t)blockIdx.x * T + threadIdx.x) * 2; i < n; i += stride) {
        double2 x, v[C];
        if (i + 1 < n) {
            x = form ? make_double2(formed(src, i, mean), formed(src, i + 1, mean)) : *reinterpret_cast<const double2*>(w + i);
            if (form && first) *reinterpret_cast<double2*>(w + i) = x;
#pragma unroll
            for (int j = 0; j < C; ++j) v[j] = *reinterpret_cast<const double2*>(col[j] + i);
        } else {
            x = make_double2(form ? formed(src, i, mean) : w[i], 0.0);
            if (form && first) w[i] = x.x;
#pragma unroll
            for (int j = 0; j < C; ++j) v[j] = make_double2(col[j][i], 0.0);
        }
        nn = fma(x.y, x.y, fma(x.x, x.x, nn));
#pragma unroll
        for (int j = 0; j < C; ++j) acc[j] = fma(v[j].y, x.y, fma(v[j].x, x.x, acc[j]));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, base = warp_sums<C>(acc, lane);
    __shared__ double sh[T / 32][C + 1];
    __shared__ double fin[T];
    sh[warp][base] = acc[0];   // lanes that share a number hold the same sum
    const bool norm = nrm && first;
    if (norm) {
        nn = warp_sum(nn);
        if (lane == 0) sh[warp][C] = nn;
    }
    __syncthreads();
    double* part = partials + (size_t)blockIdx.y * gridDim.x * (C + 1);
    if (threadIdx.x <= C && (threadIdx.x < C || norm)) {
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < T / 32; ++q) v += sh[q][threadIdx.x];
        part[(size_t)blockIdx.x * (C + 1) + threadIdx.x] = v;
    }
    if (!last_block(counter + blockIdx.y)) return;
    constexpr int G = T / C;
    const int g = threadIdx.x / C, num = threadIdx.x % C;
    double v = 0.0;
#pragma unroll 4
    for (int b = g; b < (int)gridDim.x; b += G) v += __ldcg(part + (size_t)b * (C + 1) + num);
    fin[threadIdx.x] = v;
    if (norm && warp == 0) {
        double t = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(part + (size_t)b * (C + 1) + C);
        t = warp_sum(t);
        if (lane == 0) nrm[0] = t;
    }
    __syncthreads();
    if (threadIdx.x < C && j0 + threadIdx.x < k) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < G; ++q) t += fin[q * C + threadIdx.x];
        h[j0 + threadIdx.x] = t * scale[j0 + threadIdx.x];
    }
}

// w -= sum_j h_j v_j over k = 8 a + REM columns (the remainder's loads go out together as well),
// and |w|^2 of the result.  The last block keeps the books: FIRST decides whether |w|^2 fell below
// thr times its old value (then a second pass follows); s_next = 1/|w| (0 on breakdown, which the
// host reports); host (pinned) gets the coefficients of both passes together and the norm.
template <int J>
__device__ __forceinline__ void update_columns(const double* __restrict__ p, int64_t ld, const double* c, double2& s) {
    double2 v[J > 0 ? J : 1];
#pragma unroll
    for (int j = 0; j < J; ++j) v[j] = *reinterpret_cast<const double2*>(p + (size_t)j * ld);
#pragma unroll
    for (int j = 0; j < J; ++j) {
        s.x = fma(c[j], v[j].x, s.x);
        s.y = fma(c[j], v[j].y, s.y);
    }
}
template <bool FIRST>
__device__ __forceinline__ void update_finish(double nn, int k, double* __restrict__ sc, double* __restrict__ s_next, double thr, double* host,
                                              double* __restrict__ partials, unsigned int* counter) {
    __shared__ double sh[T / 32];
    nn = warp_sum(nn);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = nn;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int q = 0; q < (int)blockDim.x / 32; ++q) v += sh[q];
        partials[blockIdx.x] = v;
    }
    if (!last_block(counter)) return;
    double v = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) v += __ldcg(partials + b);
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double tot = 0.0;
    for (int q = 0; q < (int)blockDim.x / 32; ++q) tot += sh[q];
    for (int j = threadIdx.x; j < k; j += blockDim.x) host[j] = FIRST ? sc[SC_H1 + j] : sc[SC_H1 + j] + sc[SC_H2 + j];
    if (threadIdx.x == 0) {
        if (FIRST) sc[SC_AGAIN] = tot < thr * sc[SC_NB] ? 1.0 : 0.0;
        host[SC_NA] = tot;
        s_next[0] = tot > 0.0 ? 1.0 / sqrt(tot) : 0.0;
    }
    __threadfence_system();
}
template <bool FIRST, int REM>
__global__ void __launch_bounds__(T, 4) update_kernel(const double* __restrict__ V, int64_t ld, int k, double* w, int64_t n,
                                                      double* __restrict__ sc, double* __restrict__ s_next, double thr,
                                                      double* host, double* __restrict__ partials, unsigned int* counter) {
    if (!FIRST && sc[SC_AGAIN] == 0.0) return;
    extern __shared__ double c[];   // k coefficients
    const double* h = sc + (FIRST ? SC_H1 : SC_H2);
    for (int j = threadIdx.x; j < k; j += blockDim.x) c[j] = -h[j] * sc[SC_SCALE + j];
    __syncthreads();
    double nn = 0.0;
    const int64_t pairs = (n + 1) / 2, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < pairs; q += stride) {
        const int64_t i = (pairs - 1 - q) * 2;
        const double* p = V + i;
        double2 s;
        if (i + 1 < n) {
            s = *reinterpret_cast<const double2*>(w + i);
            int j = 0;
            for (; j + 8 <= k; j += 8) update_columns<8>(p + (size_t)j * ld, ld, c + j, s);
            update_columns<REM>(p + (size_t)j * ld, ld, c + j, s);
            *reinterpret_cast<double2*>(w + i) = s;
        } else {
            s = make_double2(w[i], 0.0);
            for (int j = 0; j < k; ++j) s.x = fma(c[j], p[(size_t)j * ld], s.x);
            w[i] = s.x;
        }
        nn = fma(s.y, s.y, fma(s.x, s.x, nn));
    }
    update_finish<FIRST>(nn, k, sc, s_next, thr, host, partials, counter);
}
// The same with L lanes for an entry pair, each with every L-th column: vectors whose pairs alone leave
// the chip short of loads in flight.
template <bool FIRST, int L>
__global__ void __launch_bounds__(T, 4) update_lanes_kernel(const double* __restrict__ V, int64_t ld, int k, double* w, int64_t n,
                                                            double* __restrict__ sc, double* __restrict__ s_next, double thr,
                                                            double* host, double* __restrict__ partials, unsigned int* counter) {
    if (!FIRST && sc[SC_AGAIN] == 0.0) return;
    extern __shared__ double c[];   // coefficients, zeros up to a multiple of 8 L
    const double* h = sc + (FIRST ? SC_H1 : SC_H2);
    const int padded = (k + 8 * L - 1) / (8 * L) * (8 * L);
    for (int j = threadIdx.x; j < padded; j += T) c[j] = j < k ? -h[j] * sc[SC_SCALE + j] : 0.0;
    __syncthreads();
    double nn = 0.0;
    const int sub = threadIdx.x % L;
    const int64_t pairs = (n + 1) / 2, step = (int64_t)gridDim.x * (T / L);
    for (int64_t base = (int64_t)blockIdx.x * (T / L); base < pairs; base += step) {
        const int64_t q = base + threadIdx.x / L, i = q * 2;
        double2 s = make_double2(0.0, 0.0);
        const bool whole = i + 1 < n;
        if (q < pairs) {
            if (sub == 0) s = whole ? *reinterpret_cast<const double2*>(w + i) : make_double2(w[i], 0.0);
            const double* p = V + i;
            for (int j = sub; j < padded; j += 8 * L) {
                double2 v[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const double* a = p + (size_t)min(j + t * L, k - 1) * ld;
                    v[t] = whole ? *reinterpret_cast<const double2*>(a) : make_double2(a[0], 0.0);
                }
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    s.x = fma(c[j + t * L], v[t].x, s.x);
                    s.y = fma(c[j + t * L], v[t].y, s.y);
                }
            }
        }
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o, L);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o, L);
        }
        if (q < pairs && sub == 0) {
            if (whole) *reinterpret_cast<double2*>(w + i) = s;
            else w[i] = s.x;
            nn = fma(s.y, s.y, fma(s.x, s.x, nn));
        }
    }
    update_finish<FIRST>(nn, k, sc, s_next, thr, host, partials, counter);
}

// Short vectors, up to CLUSTER_K columns: the whole Arnoldi step in one cluster of 16 blocks, w in
// registers.  Sums cross the blocks through distributed shared memory and two cluster barriers per
// pass, where the kernels above are four launches that mostly wait.
// FP64 bound: 2 n k FMAs per pass on 16 SMs, 0.03 ns each.
namespace cg = cooperative_groups;
constexpr int CB = 16, CT = 256, CW = CT / 32, CP = 4, CLUSTER_K = 32;
constexpr int64_t CLUSTER_N = (int64_t)CB * CT * CP * 2;

__device__ __forceinline__ double2 load2(const double* p, int64_t i, int64_t n) {
    return i + 1 < n ? *reinterpret_cast<const double2*>(p + i) : make_double2(p[i], 0.0);
}
__global__ void __launch_bounds__(CT, 1) cluster_kernel(double* V, int64_t ld, int k, Source src, int64_t n, double* __restrict__ sc,
                                                        double thr, double* host) {
    __shared__ double part[CW][CLUSTER_K + 1];   // sums of each warp: column j, then |w|^2
    // of the block, per pass, read by the whole cluster: the columns, |w|^2 before the pass behind them
    // (first pass) and after it in a slot of its own.  Nothing but a block barrier lies between the
    // reads of the first two and the write of the last, so no column count may share a slot with it.
    constexpr int AFTER = CLUSTER_K + 1;
    __shared__ double blk[2][AFTER + 1];
    __shared__ double fin[4][64], c[CLUSTER_K], nrm[2][CW], bn[2];
    cg::cluster_group cl = cg::this_cluster();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t pairs = (n + 1) / 2, q0 = (int64_t)blockIdx.x * CT + threadIdx.x;
    const bool busy = q0 - lane < pairs;   // the warp has entries at all (P = 0 then for some lanes)
    double* w = V + (size_t)k * ld;
    double2 x[CP];
    int64_t at[CP];
    const double mean = src.mean ? src.a * src.mean[0] : 0.0;
    double before = 0.0;
#pragma unroll
    for (int p = 0; p < CP; ++p) {
        const int64_t q = q0 + (int64_t)p * (CB * CT);
        at[p] = q < pairs ? 2 * q : -1;
        x[p] = make_double2(0.0, 0.0);
        if (at[p] >= 0) {
            if (src.yf || src.yd) x[p] = make_double2(formed(src, at[p], mean), at[p] + 1 < n ? formed(src, at[p] + 1, mean) : 0.0);
            else x[p] = load2(w, at[p], n);
        }
        before = fma(x[p].y, x[p].y, fma(x[p].x, x[p].x, before));
    }
    double tot = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        if (busy) {
            for (int j0 = 0; j0 < k; j0 += 8) {
                double acc[8];
#pragma unroll
                for (int t = 0; t < 8; ++t) acc[t] = 0.0;
#pragma unroll
                for (int p = 0; p < CP; ++p) {
                    if (at[p] < 0) break;
                    double2 v[8];
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        if (j0 + t < k) v[t] = load2(V + (size_t)(j0 + t) * ld, at[p], n);
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        if (j0 + t < k) acc[t] = fma(v[t].y, x[p].y, fma(v[t].x, x[p].x, acc[t]));
                }
                __syncwarp();
                const int j = j0 + warp_sums<8>(acc, lane);
                if (j < k) part[warp][j] = acc[0];   // lanes that share a number hold the same sum
            }
            if (pass == 0) {
                before = warp_sum(before);
                if (lane == 0) part[warp][k] = before;
            }
        } else {
            for (int j = lane; j <= k; j += 32) part[warp][j] = 0.0;
        }
        __syncthreads();
        const int cols = k + (pass == 0 ? 1 : 0);
        if (threadIdx.x < cols) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < CW; ++q) s += part[q][threadIdx.x];
            blk[pass][threadIdx.x] = s;
        }
        cl.sync();
        // four groups of 64 threads, one per column, take four blocks each
        {
            static_assert(CLUSTER_K + 1 <= 64 && CT == 256, "a thread of a group per column");
            const int g = threadIdx.x >> 6, j = threadIdx.x & 63;
            double s = 0.0;
            if (j < cols)
#pragma unroll
                for (int b = 0; b < CB / 4; ++b) s += *cl.map_shared_rank(&blk[pass][j], g * (CB / 4) + b);
            fin[g][j] = s;
            __syncthreads();
            if (g == 0 && j < cols) {
                s = (fin[0][j] + fin[1][j]) + (fin[2][j] + fin[3][j]);
                if (j < k) {
                    const double sj = sc[SC_SCALE + j], h = s * sj;
                    c[j] = -h * sj;
                    if (blockIdx.x == 0) {
                        if (pass == 0) sc[SC_H1 + j] = h;
                        host[j] = pass == 0 ? h : sc[SC_H1 + j] + h;
                    }
                } else {
                    bn[0] = s;   // |w|^2 before
                }
            }
            __syncthreads();
        }
        double nn = 0.0;
#pragma unroll
        for (int p = 0; p < CP; ++p) {
            if (at[p] < 0) break;
            double2 s = x[p];
            for (int j0 = 0; j0 < k; j0 += 8) {
                double2 v[8];
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (j0 + t < k) v[t] = load2(V + (size_t)(j0 + t) * ld, at[p], n);
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (j0 + t < k) {
                        s.x = fma(c[j0 + t], v[t].x, s.x);
                        s.y = fma(c[j0 + t], v[t].y, s.y);
                    }
            }
            x[p] = s;
            nn = fma(s.y, s.y, fma(s.x, s.x, nn));
        }
        __syncwarp();
        if (busy) nn = warp_sum(nn);
        if (lane == 0) nrm[pass][warp] = nn;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < CW; ++q) s += nrm[pass][q];
            blk[pass][AFTER] = s;
        }
        cl.sync();
        if (warp == 0) {
            double s = lane < CB ? *cl.map_shared_rank(&blk[pass][AFTER], lane) : 0.0;
#pragma unroll
            for (int o = CB / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) bn[1] = s;
        }
        __syncthreads();
        tot = bn[1];
        if (!(tot < thr * bn[0])) break;   // the same numbers in every block: all leave together
    }
#pragma unroll
    for (int p = 0; p < CP; ++p) {
        if (at[p] < 0) break;
        if (at[p] + 1 < n) *reinterpret_cast<double2*>(w + at[p]) = x[p];
        else w[at[p]] = x[p].x;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        host[SC_NA] = tot;
        sc[SC_SCALE + k] = tot > 0.0 ? 1.0 / sqrt(tot) : 0.0;
    }
    __threadfence_system();
    cl.sync();   // no block leaves while its sums may still be read
}
cudaError_t launch_cluster(double* V, int64_t ld, int k, const Source& src, int64_t n, double* sc, double thr, double* host,
                           cudaStream_t st) {
    // more than 8 blocks are a cluster only where the kernel allows it, on this device
    const cudaError_t allowed = cudaFuncSetAttribute(cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (allowed != cudaSuccess) return allowed;
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeClusterDimension;
    a.val.clusterDim = {CB, 1, 1};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CB);
    cfg.blockDim = dim3(CT);
    cfg.stream = st;
    cfg.attrs = &a;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, cluster_kernel, V, ld, k, src, n, sc, thr, host);
}

// u = sum_{j<k} y_j v_j
__global__ void combine_kernel(const double* __restrict__ V, int64_t ld, int k, const double* __restrict__ y,
                               const double* __restrict__ scale, double* __restrict__ u, int64_t n) {
    extern __shared__ double c[];
    for (int j = threadIdx.x; j < k; j += blockDim.x) c[j] = y[j] * scale[j];
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double s = 0.0;
#pragma unroll 4
        for (int j = 0; j < k; ++j) s = fma(c[j], V[(size_t)j * ld + i], s);
        u[i] = s;
    }
}

constexpr int CC = COLUMNS / COUNTERS;
template <bool FIRST>
void launch_update(int lanes, int nu, const double* V, int64_t ld, int k, double* w, int64_t n, double* sc, double* sk, double thr,
                   double* host, double* partials, unsigned int* counter, cudaStream_t st) {
    const size_t sh = (size_t)(k + 8 * lanes) * sizeof(double);
    switch (lanes > 1 ? 8 + lanes : k % 8) {
#define CHNS_UPDATE(R) case R: update_kernel<FIRST, R><<<nu, T, sh, st>>>(V, ld, k, w, n, sc, sk, thr, host, partials, counter); break
#define CHNS_LANES(L) case 8 + L: update_lanes_kernel<FIRST, L><<<nu, T, sh, st>>>(V, ld, k, w, n, sc, sk, thr, host, partials, counter); break
        CHNS_UPDATE(0); CHNS_UPDATE(1); CHNS_UPDATE(2); CHNS_UPDATE(3);
        CHNS_UPDATE(4); CHNS_UPDATE(5); CHNS_UPDATE(6); CHNS_UPDATE(7);
        CHNS_LANES(2); CHNS_LANES(4); CHNS_LANES(8);
#undef CHNS_LANES
#undef CHNS_UPDATE
    }
}
template <int K = 32>
void launch_dots(int kk, int nb, const double* V, int64_t ld, const Source& s, double* w, int64_t n, const double* scale, double* h,
                 double* nrm, double* partials, unsigned int* counter, const double* pred, cudaStream_t st) {
    if (kk == K) dots_kernel<K><<<nb, T, 0, st>>>(V, ld, s, w, n, scale, h, nrm, partials, counter, pred);
    else if constexpr (K > 1) launch_dots<K - 1>(kk, nb, V, ld, s, w, n, scale, h, nrm, partials, counter, pred, st);
}
}  // namespace

// Which split.  All of an Arnoldi step, us, mean over 1..30 / 1..60 / 1..120 / 1..250 columns (one pass each):
//   n            long-vector kernels      chunks                   cluster
//   5,445        36 /  53 /  96 / 140     33 / 34 / 39 / 42        23 / 34 /  63 /  93
//   21,125       34 /  46 /  68 / 116     31 / 33 / 37 / 45        32 / 48 /  77 / 138
//   34,105       34 /  47 /  69 / 118     33 / 36 / 40 / 49
//   83,205       43 /  61 /  97 / 176     39 / 46 / 60 / 93
//   215,622      70 / 102 / 167 / 286     60 / 77 / 111 / 189
//   487,302      72 / 113 / 198 / 381     70 / 102 / 165 / 305
//   1,315,845    124 / 209 / 380 / 750    135 / 219 / 387 / 758
// The cluster wins while its 16 SMs have little to do: up to 32 columns, and n k up to 300,000 (13,605
// values: 23 columns, 21,125: 15, 29,478: 10), 14 to 24 us per step against 27 to 33.
constexpr int64_t CLUSTER_NK = 300000, CHUNKS_N = 1 << 19;   // 2^19: between the last two rows
int orthogonalise(double* V, int64_t ld, int k, const Source& src, int64_t n, double* sc, double thr, double* host, double* partials,
                  unsigned int* counter, cudaStream_t st) {
    if (n <= CLUSTER_N && k <= CLUSTER_K && n * k <= CLUSTER_NK) {
        if (launch_cluster(V, ld, k, src, n, sc, thr, host, st) == cudaSuccess) return 1;
        (void)cudaGetLastError();   // no room for the cluster (a partitioned device): the general kernels
    }
    const int64_t sms = chns_num_sms(), pairs = (n + 1) / 2, need = (n + 2 * T - 1) / (2 * T);
    const bool chunked = n < CHUNKS_N;
    Source in_place = src;
    in_place.yf = nullptr, in_place.yd = nullptr, in_place.mean = nullptr;
    double *w = V + (size_t)k * ld, *sk = sc + SC_SCALE + k;
    // lanes per pair of the update: as many as leave no thread a second pair (250 columns on 5,445 values: 67 us
    // a step with one lane, 42 with eight; 46,014: 61, 62; 13,605: 55, 40, and 38 with four)
    int lanes = chunked ? 8 : 1, nk = 0;
    while (lanes > 1 && pairs * lanes > T * sms) lanes /= 2;
    const int nu = (int)std::min(lanes > 1 ? (pairs * lanes + T - 1) / T : need, 4 * sms);
    for (bool first : {true, false}) {
        double *h = sc + (first ? SC_H1 : SC_H2), *nrm = first ? sc + SC_NB : nullptr;
        const double* pred = first ? nullptr : sc + SC_AGAIN;
        if (chunked) {
            const int64_t chunks = (k + CC - 1) / CC;
            const dim3 nb((unsigned)std::max<int64_t>(1, std::min(need, 2 * sms / chunks)), (unsigned)chunks);
            dots_chunks_kernel<CC><<<nb, T, 0, st>>>(V, ld, k, first ? src : in_place, w, n, sc + SC_SCALE, h, nrm, partials, counter, pred);
            ++nk;
        } else {
            for (int j0 = 0; j0 < k; j0 += 32, ++nk)
                launch_dots(std::min(k - j0, 32), (int)std::min(need, 2 * sms), V + (size_t)j0 * ld, ld, first && j0 == 0 ? src : in_place, w, n,
                            sc + SC_SCALE + j0, h + j0, j0 == 0 ? nrm : nullptr, partials, counter, pred, st);
        }
        if (first) launch_update<true>(lanes, nu, V, ld, k, w, n, sc, sk, thr, host, partials, counter, st);
        else launch_update<false>(lanes, nu, V, ld, k, w, n, sc, sk, thr, host, partials, counter, st);
        ++nk;
    }
    return nk;
}
void combine(const double* V, int64_t ld, int k, const double* y, const double* scale, double* u, int64_t n, cudaStream_t st) {
    const int64_t need = (n + T - 1) / T, cap = 8 * (int64_t)chns_num_sms();
    combine_kernel<<<(unsigned)std::min(need, cap), T, k * sizeof(double), st>>>(V, ld, k, y, scale, u, n);
}

}  // namespace krylov
