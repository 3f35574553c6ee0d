// Vector kernels of the Arnoldi process (Newton's GMRES and the adjoint's), FP64.
//
// The basis is kept unnormalised: slot j of V holds w_j and a device scalar s_j = 1/|w_j|, and
// v_j = s_j w_j.  The scale rides along where a vector is read anyway, so no pass normalises.
// One Gram-Schmidt pass is a dot kernel (32 columns at a time, forming w = S y + mean on the way)
// and an update kernel with the new norm; the last block of each sums the partials, in a fixed
// order, and the update's writes what the host waits for into pinned memory.  A second pass is
// queued behind the first and decided on the device: its blocks return at once when |w| kept a
// tenth of its length.  (Left to the host, it costs a discarded operator application whenever it
// is wanted, which is often: two drops, 81 -> 118 ms per Newton step.)
//
// Bound: k FP64 FMAs per entry and pass on the narrow FP64 pipe (n = 1.65 M, k = 15: 39 us) next
// to one read of V (29 us).  The kernels are instantiated per number of columns (dots) or per
// remainder (update), so that all loads of an entry pair go out together, and few threads take many
// rows, so that the reductions add 5 % of FP64 work instead of the 60 % of eight columns per
// thread.  The update walks the rows backwards, where the dot pass has just left its columns in L2
// (evict-first loads there: 34 -> 50 us).
//   n = 1.65 M, k = 1..30: dots 3.3 us per column + 24 us (w formed, 4 us of reduction), update
//   2.7 us per column + 10 us; all of an Arnoldi step's vector work 181 -> 136 us, and without the
//   33 us of the normalising, scaling and mean passes that it takes in.
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

// Short vectors: the whole Arnoldi step in one cluster of 16 blocks, w in registers.  Sums cross the
// blocks through distributed shared memory and two cluster barriers per pass, where the kernels above
// are four launches (six and more from 33 columns on) of 6 to 10 us that mostly wait.
//   n = 5,445 (2D), 20 columns on average: 35 -> 20 us per Arnoldi step; n = 4,374 (3D), 60 columns
//   and two passes: 26 us.  FP64 bound: 2 n k FMAs per pass on 16 SMs, 0.03 ns each.
namespace cg = cooperative_groups;
constexpr int CB = 16, CT = 256, CW = CT / 32, CP = 4;
constexpr int64_t CLUSTER_N = (int64_t)CB * CT * CP * 2;

__device__ __forceinline__ double2 load2(const double* p, int64_t i, int64_t n) {
    return i + 1 < n ? *reinterpret_cast<const double2*>(p + i) : make_double2(p[i], 0.0);
}
__global__ void __launch_bounds__(CT, 1) cluster_kernel(double* V, int64_t ld, int k, Source src, int64_t n, double* __restrict__ sc,
                                                        double thr, double* host) {
    __shared__ double part[CW][257];   // sums of each warp: column j, then |w|^2
    // of the block, per pass, read by the whole cluster: up to 256 columns, |w|^2 before the pass behind
    // them (first pass) and after it in a slot of its own.  Nothing but a block barrier lies between the
    // reads of the first two and the write of the last, so no column count may share a slot with it.
    constexpr int AFTER = 257;
    __shared__ double blk[2][AFTER + 1];
    __shared__ double fin[4][64], c[256], nrm[2][CW], bn[2];
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
        for (int j = threadIdx.x; j < cols; j += CT) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < CW; ++q) s += part[q][j];
            blk[pass][j] = s;
        }
        cl.sync();
        // four groups of threads take four blocks each, 64 columns at a time
        for (int j0 = 0; j0 < cols; j0 += 64) {
            const int g = threadIdx.x >> 6, j = j0 + (threadIdx.x & 63);
            double s = 0.0;
            if (j < cols)
#pragma unroll
                for (int b = 0; b < CB / 4; ++b) s += *cl.map_shared_rank(&blk[pass][j], g * (CB / 4) + b);
            fin[g][threadIdx.x & 63] = s;
            __syncthreads();
            if (threadIdx.x < 64 && j < cols) {
                s = (fin[0][threadIdx.x] + fin[1][threadIdx.x]) + (fin[2][threadIdx.x] + fin[3][threadIdx.x]);
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

template <bool FIRST>
void launch_update(int nu, int th, const double* V, int64_t ld, int k, double* w, int64_t n, double* sc, double* sk, double thr,
                   double* host, double* partials, unsigned int* counter, cudaStream_t st) {
    const size_t sh = k * sizeof(double);
    switch (k % 8) {
#define CHNS_UPDATE(R) case R: update_kernel<FIRST, R><<<nu, th, sh, st>>>(V, ld, k, w, n, sc, sk, thr, host, partials, counter); break
        CHNS_UPDATE(0); CHNS_UPDATE(1); CHNS_UPDATE(2); CHNS_UPDATE(3);
        CHNS_UPDATE(4); CHNS_UPDATE(5); CHNS_UPDATE(6); CHNS_UPDATE(7);
#undef CHNS_UPDATE
    }
}
template <int K = 32>
void launch_dots(int kk, int nb, int th, const double* V, int64_t ld, const Source& s, double* w, int64_t n, const double* scale,
                 double* h, double* nrm, double* partials, unsigned int* counter, const double* pred, cudaStream_t st) {
    if (kk == K) dots_kernel<K><<<nb, th, 0, st>>>(V, ld, s, w, n, scale, h, nrm, partials, counter, pred);
    else if constexpr (K > 1) launch_dots<K - 1>(kk, nb, th, V, ld, s, w, n, scale, h, nrm, partials, counter, pred, st);
}
}  // namespace

int orthogonalise(double* V, int64_t ld, int k, const Source& src, int64_t n, double* sc, double thr, double* host, double* partials,
                  unsigned int* counter, cudaStream_t st) {
    // one cluster: 16 of the SMs, so only while their FP64 pipes are quicker than four launches.
    // Arnoldi step at 20 and 40 columns: n = 5,445: 25, 34 us against 41, 56; 15,765: 30, 44 against
    // 46, 68; 29,478: 46, 72 against 57, 87 (both sides grow with n k from there)
    if (n <= CLUSTER_N) {
        if (launch_cluster(V, ld, k, src, n, sc, thr, host, st) == cudaSuccess) return 1;
        (void)cudaGetLastError();   // no room for the cluster (a partitioned device): the general kernels
    }
    // small vectors take two-warp blocks: the reductions are FP64 work per block, and the FP64 pipe
    // is per SM
    const int64_t sms = chns_num_sms();
    const int th = n < 256 * sms ? 64 : T;
    const int64_t need = (n + 2 * th - 1) / (2 * th);
    const int nb = (int)std::min<int64_t>(need, 2 * (T / th) * sms);
    const int nu = (int)std::min<int64_t>(need, 4 * (T / th) * sms);
    double* w = V + (size_t)k * ld;
    int nk = 0;
    for (bool first : {true, false}) {
        for (int j0 = 0; j0 < k; j0 += 32) {
            Source s = src;
            const bool form = first && j0 == 0;
            if (!form) s.yf = nullptr, s.yd = nullptr, s.mean = nullptr;
            launch_dots(std::min(k - j0, 32), nb, th, V + (size_t)j0 * ld, ld, s, w, n, sc + SC_SCALE + j0,
                        sc + (first ? SC_H1 : SC_H2) + j0, form ? sc + SC_NB : nullptr, partials, counter,
                        first ? nullptr : sc + SC_AGAIN, st);
            ++nk;
        }
        double* sk = sc + SC_SCALE + k;
        if (first) launch_update<true>(nu, th, V, ld, k, w, n, sc, sk, thr, host, partials, counter, st);
        else launch_update<false>(nu, th, V, ld, k, w, n, sc, sk, thr, host, partials, counter, st);
        ++nk;
    }
    return nk;
}
void combine(const double* V, int64_t ld, int k, const double* y, const double* scale, double* u, int64_t n, cudaStream_t st) {
    const int64_t need = (n + T - 1) / T, cap = 8 * (int64_t)chns_num_sms();
    combine_kernel<<<(unsigned)std::min(need, cap), T, k * sizeof(double), st>>>(V, ld, k, y, scale, u, n);
}

}  // namespace krylov
