// Newton's method of Section 3.4, matrix-free: each Newton iteration solves
// J dU = -R (Eq. newton_linear_system) with right-preconditioned restarted GMRES whose
// operator is the J x element kernel (FP32 in mixed mode, FP64 otherwise) and whose
// preconditioner is nodal block-Jacobi (plus the pressure Schur and Cahn-Hilliard
// blocks); orthogonalisation (classical Gram-Schmidt with selective re-orthogonalisation),
// dots, norms, the residual and the update stay FP64 on the device.  With the pressure
// level set by its mean (pin mode 2) J is singular (constant pressure); GMRES runs on
// J + u m_p^T / |Omega| instead, which is nonsingular and has the zero-mean solution of
// J dU = -R.  Gram-Schmidt (including the decision to re-orthogonalise) and the next
// Arnoldi vector stay on the device; the Hessenberg column goes to the host for the
// Givens update, and that read-back overlaps the next vector's operator application,
// which is queued before the host waits.
#include <cuda_runtime.h>

#include <cmath>
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <utility>
#include <vector>

#include "block_jacobi.h"
#include "chns_internal.h"
#include "krylov.h"
#include "precond.h"
#include "reduce.cuh"

struct SolverWS {
    int restart = 0;
    int64_t n = 0, N = 0, ld = 0;
    double* V = nullptr;     // (restart + 1) * ld Arnoldi basis (ld: n rounded up to 16 bytes)
    double* w = nullptr;     // n
    double* R = nullptr;     // n residual
    double* dU = nullptr;    // n Newton update
    double* z64 = nullptr;   // n
    double* t64 = nullptr;   // n
    double* S = nullptr;     // n row scaling 1/|diag J| of the current linearisation
    double* Sd = nullptr;    // n its inverse |diag J| (identity rows: 1)
    double* S0 = nullptr;    // n row scaling of the first Newton iterate (norm of the step)
    double* SR = nullptr;    // n scaled residual
    float* Uo32 = nullptr;   // n
    float* Us32 = nullptr;   // n
    float* z32 = nullptr;    // n
    float* y32 = nullptr;    // n
    float* Pblk32 = nullptr; // N * nf * nf block diagonal (FP32 build)
    double* Pblk64 = nullptr;
    float* Pinv32 = nullptr; // inverted blocks
    double* Pinv64 = nullptr;
    double* sc = nullptr;    // device scalars
    double* hsc = nullptr;   // pinned host scalars
    cudaEvent_t ev[16] = {};  // J x, preconditioner build / apply and Gram-Schmidt timing (two sets
                              // of J x / apply events alternate between Arnoldi steps)
    float* ce = nullptr;     // E element coefficients of the pressure Schur approximation
    double* part = nullptr;  // per-block partials of the Gram-Schmidt reductions
    double* mpart = nullptr; // and of the pressure mean
    unsigned int* counter = nullptr;   // blocks that finished: Gram-Schmidt (krylov::COUNTERS), pressure mean
    float* ch_psi2 = nullptr;  // psi''(phi~) at the nodes (Cahn-Hilliard block)
};

void chns_solver_ws_free(SolverWS* ws) {
    if (!ws) return;
    cudaFree(ws->V);
    cudaFree(ws->w);
    cudaFree(ws->R);
    cudaFree(ws->dU);
    cudaFree(ws->z64);
    cudaFree(ws->t64);
    cudaFree(ws->S);
    cudaFree(ws->Sd);
    cudaFree(ws->S0);
    cudaFree(ws->SR);
    cudaFree(ws->Uo32);
    cudaFree(ws->Us32);
    cudaFree(ws->z32);
    cudaFree(ws->y32);
    cudaFree(ws->Pblk32);
    cudaFree(ws->Pblk64);
    cudaFree(ws->Pinv32);
    cudaFree(ws->Pinv64);
    cudaFree(ws->sc);
    cudaFree(ws->ce);
    cudaFree(ws->part);
    cudaFree(ws->mpart);
    cudaFree(ws->counter);
    cudaFree(ws->ch_psi2);
    if (ws->hsc) cudaFreeHost(ws->hsc);
    for (auto& e : ws->ev)
        if (e) cudaEventDestroy(e);
    delete ws;
}

namespace {

constexpr int MAXSC = 1024;

chns_status ensure_ws(chns_mesh* m, int restart) {
    SolverWS* ws = m->ws;
    if (ws && ws->restart >= restart) return CHNS_OK;
    if (ws) {
        precond_drop_graphs(m);   // they hold the old workspace's vectors
        chns_solver_ws_free(ws);
    }
    m->ws = nullptr;
    ws = new SolverWS();
    ws->restart = restart;
    ws->N = m->dm.N;
    ws->n = m->dm.N * m->dm.nf;
    ws->ld = (ws->n + 1) / 2 * 2;
    const size_t n = (size_t)ws->n, nb = (size_t)m->dm.N * m->dm.nf * m->dm.nf;
    cudaError_t e = cudaSuccess;
    auto A = [&](void** p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    };
    A((void**)&ws->V, (size_t)(restart + 1) * ws->ld * sizeof(double));
    A((void**)&ws->w, n * sizeof(double));
    A((void**)&ws->R, n * sizeof(double));
    A((void**)&ws->dU, n * sizeof(double));
    A((void**)&ws->z64, n * sizeof(double));
    A((void**)&ws->t64, n * sizeof(double));
    A((void**)&ws->S, n * sizeof(double));
    A((void**)&ws->Sd, n * sizeof(double));
    A((void**)&ws->S0, n * sizeof(double));
    A((void**)&ws->SR, n * sizeof(double));
    A((void**)&ws->Uo32, n * sizeof(float));
    A((void**)&ws->Us32, n * sizeof(float));
    A((void**)&ws->z32, n * sizeof(float));
    A((void**)&ws->y32, n * sizeof(float));
    A((void**)&ws->Pblk32, nb * sizeof(float));
    A((void**)&ws->Pblk64, nb * sizeof(double));
    A((void**)&ws->Pinv32, nb * sizeof(float));
    A((void**)&ws->Pinv64, nb * sizeof(double));
    A((void**)&ws->sc, MAXSC * sizeof(double));
    A((void**)&ws->ce, (size_t)m->dm.E * sizeof(float));
    A((void**)&ws->part, (size_t)33 * 4 * std::max(chns_num_sms(), 8) * sizeof(double));   // 33 numbers of up to 4 blocks per SM
    A((void**)&ws->mpart, (size_t)(m->dm.N / 64 + 64) * sizeof(double));
    A((void**)&ws->counter, (krylov::COUNTERS + 1) * sizeof(unsigned int));
    if (e == cudaSuccess) e = cudaMemset(ws->counter, 0, (krylov::COUNTERS + 1) * sizeof(unsigned int));
    A((void**)&ws->ch_psi2, (size_t)m->dm.N * sizeof(float));
    if (e == cudaSuccess) e = cudaMallocHost((void**)&ws->hsc, MAXSC * sizeof(double));
    for (auto& ev : ws->ev)
        if (e == cudaSuccess) e = cudaEventCreate(&ev);
    if (e != cudaSuccess) {
        chns_solver_ws_free(ws);
        return chns_cuda_status(e, "cudaMalloc(solver workspace)");
    }
    m->ws = ws;
    return CHNS_OK;
}

// ---------------- BLAS-1 ----------------
__global__ void copy64_kernel(const double* __restrict__ a, double* __restrict__ b, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = a[i];
}
__global__ void to32_kernel(const double* __restrict__ a, float* __restrict__ b, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}
__global__ void to64_kernel(const float* __restrict__ a, double* __restrict__ b, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (double)a[i];
}
// sum_n m_n (a + b - c)[n*NF + f] into per-block partials (the phi-mass change of a
// Newton update: a = U, b = dU, c = U^k)
__global__ void field_mass3_kernel(const double* __restrict__ m, const double* __restrict__ a,
                                   const double* __restrict__ b, const double* __restrict__ c, int NF, int f,
                                   int64_t N, double* partials) {
    double acc[1] = {0.0};
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x) {
        const size_t i = (size_t)n * NF + f;
        acc[0] += m[n] * ((a[i] + b[i]) - c[i]);
    }
    block_reduce_store<1>(acc, partials);
}
// y = a s .* x
template <class T>
__global__ void scale_vec_kernel(const T* x, const double* __restrict__ sv, double* y, double a, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = a * (sv[i] * (double)x[i]);
}
__global__ void axpy_kernel(double a, const double* __restrict__ x, double* __restrict__ y, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] += a * x[i];
}
// y = a*x + b*y
__global__ void axpby_kernel(double a, const double* __restrict__ x, double b, double* __restrict__ y, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = a * x[i] + b * y[i];
}

int grid_for(int64_t n) {
    int64_t b = (n + 255) / 256;
    const int64_t cap = 8 * (int64_t)chns_num_sms();
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

// ---------------- block-Jacobi preconditioner ----------------
// Replace Dirichlet / pin rows by identity rows and invert every block (Gauss-Jordan
// with partial pivoting in FP64).
template <class TB, class TI>
__global__ void pc_invert_kernel(DevMesh m, const TB* __restrict__ blk, TI* __restrict__ inv, int pin,
                                 double* __restrict__ scale, double* __restrict__ unscale, int decouple_p) {
    const int NF = m.nf, D = m.dim;
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= m.N) return;
    double A[6][12];
    for (int i = 0; i < NF; ++i)
        for (int j = 0; j < NF; ++j) {
            A[i][j] = (double)blk[((size_t)n * NF + i) * NF + j];
            A[i][NF + j] = (i == j) ? 1.0 : 0.0;
        }
    const unsigned fl = m.nflag[n];
    for (int i = 0; i < NF; ++i) {
        const bool idrow = (i < D && ((fl >> i) & 1u)) || (i == D && pin == 1 && n == 0);
        if (idrow)
            for (int j = 0; j < NF; ++j) A[i][j] = (i == j) ? 1.0 : 0.0;
    }
    // row equilibration 1/|J_ii| (identity rows: 1)
    for (int i = 0; i < NF; ++i) {
        const double a = fabs(A[i][i]);
        scale[(size_t)n * NF + i] = a > 1e-300 ? 1.0 / a : 1.0;
        if (unscale) unscale[(size_t)n * NF + i] = a > 1e-300 ? a : 1.0;
    }
    if (decouple_p & 1) {
        // the pressure is preconditioned separately (Schur-complement approximation)
        for (int j = 0; j < NF; ++j) A[D][j] = A[j][D] = (j == D) ? 1.0 : 0.0;
    }
    if (decouple_p & 2) {
        // phi and mu are preconditioned by the Cahn-Hilliard block solve
        for (int i = D + 1; i < NF; ++i)
            for (int j = 0; j < NF; ++j) A[i][j] = A[j][i] = (j == i) ? 1.0 : 0.0;
    }
    for (int col = 0; col < NF; ++col) {
        int piv = col;
        for (int r = col + 1; r < NF; ++r)
            if (fabs(A[r][col]) > fabs(A[piv][col])) piv = r;
        if (piv != col)
            for (int j = 0; j < 2 * NF; ++j) {
                const double tmp = A[col][j];
                A[col][j] = A[piv][j];
                A[piv][j] = tmp;
            }
        double d = A[col][col];
        if (d == 0.0) d = 1e-300;
        const double inv_d = 1.0 / d;
        for (int j = 0; j < 2 * NF; ++j) A[col][j] *= inv_d;
        for (int r = 0; r < NF; ++r) {
            if (r == col) continue;
            const double f = A[r][col];
            if (f != 0.0)
                for (int j = 0; j < 2 * NF; ++j) A[r][j] -= f * A[col][j];
        }
    }
    for (int i = 0; i < NF; ++i)
        for (int j = 0; j < NF; ++j) inv[((size_t)n * NF + i) * NF + j] = (TI)A[i][NF + j];
}

// First part of a preconditioner application: x = scale * v .* Sd (either may be null), z = P^{-1} x
// with the nodal blocks (P^{-T}: TRANS) in the precision they are stored in, and the rows that are
// preconditioned as scalar operators (mask 1: p; 2: phi, mu) to their compact FP32 inputs instead.
// One thread per row: the n_f entries of a row of blocks are read by its thread, neighbouring rows
// by neighbouring threads.  (64^3, FP32: 15 us; one thread per node, behind a pass that scaled v:
// 6.8 + 25.6 us.)
constexpr int PC_NODES = 32;
template <int NF, bool TRANS, class TI, class TO>
__global__ void __launch_bounds__(PC_NODES * NF) pc_first_kernel(int64_t N, int mask, const TI* __restrict__ inv,
                                                                 const double* __restrict__ v,
                                                                 const double* __restrict__ scale,
                                                                 const double* __restrict__ Sd, TO* __restrict__ z,
                                                                 PrecondIn in) {
    constexpr int D = NF - 3;
    __shared__ TI xs[PC_NODES * NF];
    __shared__ TI bl[TRANS ? PC_NODES * NF * NF : 1];
    const int64_t node0 = (int64_t)blockIdx.x * PC_NODES;
    const int ln = threadIdx.x / NF, row = threadIdx.x % NF;
    const int64_t node = node0 + ln, i = node0 * NF + threadIdx.x;
    const bool ok = node < N;
    double x = 0.0;
    if (ok) {
        x = v[i];
        if (scale) x *= scale[0];
        if (Sd) x *= Sd[i];
    }
    xs[threadIdx.x] = (TI)x;
    if (TRANS) {
        const int64_t end = N * NF * NF;
        for (int t = threadIdx.x; t < PC_NODES * NF * NF; t += PC_NODES * NF)
            bl[t] = node0 * NF * NF + t < end ? inv[node0 * NF * NF + t] : TI(0);
    }
    __syncthreads();
    if (!ok) return;
    if (row == D && (mask & 1)) {
        in.p[node] = (float)x;
        return;
    }
    if (row > D && (mask & 2)) {
        (row == D + 1 ? in.phi : in.mu)[node] = (float)x;
        return;
    }
    TI s = TI(0);
#pragma unroll
    for (int j = 0; j < NF; ++j) {
        const TI a = TRANS ? bl[(ln * NF + j) * NF + row] : inv[(size_t)i * NF + j];
        s += a * xs[ln * NF + j];
    }
    z[i] = (TO)s;
}
template <bool TRANS, class TI, class TO>
void launch_pc_first(const chns_mesh* m, int mask, const TI* inv, const double* v, const double* scale, const double* Sd, TO* z,
                     cudaStream_t s) {
    const int64_t N = m->dm.N;
    const unsigned g = (unsigned)((N + PC_NODES - 1) / PC_NODES);
    const PrecondIn in = mask ? precond_inputs(m) : PrecondIn();
    if (m->dm.nf == 5) pc_first_kernel<5, TRANS, TI, TO><<<g, PC_NODES * 5, 0, s>>>(N, mask, inv, v, scale, Sd, z, in);
    else pc_first_kernel<6, TRANS, TI, TO><<<g, PC_NODES * 6, 0, s>>>(N, mask, inv, v, scale, Sd, z, in);
    chns_count_launches(1);
}
__global__ void set_scalar_kernel(double* p, double v) { *p = v; }

// sum_n m_n v[n*NF + f] into per-block partials
template <class T>
__global__ void field_mass_kernel(const double* __restrict__ m, const T* __restrict__ v, int NF, int f,
                                  int64_t N, double* partials) {
    double acc[1] = {0.0};
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x)
        acc[0] += m[n] * (double)v[(size_t)n * NF + f];
    block_reduce_store<1>(acc, partials);
}
// y = sv .* x + a * sc[0] on the rows of field f: the scaled operator of
// J' = J + u m_p^T / |Omega| (pin mode 2), u = |diag J| on the pressure rows, so S u = 1
// there.  The rank-one term moves the null mode of J (constant pressure) off zero.
template <class T>
__global__ void scale_vec_pmean_kernel(const T* x, const double* __restrict__ sv, double* y,
                                       int64_t n, int NF, int f, const double* __restrict__ sc, double a) {
    const double s = a * sc[0];
    const int64_t N = n / NF;
    for (int64_t node = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; node < N;
         node += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i0 = node * NF;
        for (int g = 0; g < NF; ++g) y[i0 + g] = sv[i0 + g] * (double)x[i0 + g] + (g == f ? s : 0.0);
    }
}
// v[n*NF + f] -= sc[0] * inv_vol
__global__ void field_shift_kernel(double* __restrict__ v, int NF, int f, int64_t N, const double* __restrict__ sc,
                                   double inv_vol) {
    const double s = sc[0] * inv_vol;
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x)
        v[(size_t)n * NF + f] -= s;
}
struct Ctx {
    chns_mesh* m;
    SolverWS* ws;
    cudaStream_t s;
    int64_t n;
    int g;
};

// host read of k device scalars (synchronises)
chns_status read_sc(Ctx& c, const double* dev, int k, double* host) {
    CHNS_CUDA(cudaMemcpyAsync(c.ws->hsc, dev, k * sizeof(double), cudaMemcpyDeviceToHost, c.s));
    CHNS_CUDA(cudaStreamSynchronize(c.s));
    std::memcpy(host, c.ws->hsc, k * sizeof(double));
    return CHNS_OK;
}

chns_status dot_host(Ctx& c, const double* a, const double* b, double* out) {
    CHNS_CUDA(launch_dot(c.m, a, b, c.n, c.ws->sc, c.s));
    return read_sc(c, c.ws->sc, 1, out);
}

// nodal psi''(phi~) with phi~ the mid-point average (FP32)
template <class T>
__global__ void ch_nodal_kernel(int64_t N, int NF, int fphi, const T* __restrict__ Uo, const T* __restrict__ Un,
                                float* __restrict__ psi2) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const float ph = 0.5f * ((float)Uo[(size_t)n * NF + fphi] + (float)Un[(size_t)n * NF + fphi]);
    psi2[n] = 3.0f * ph * ph - 1.0f;
}

// What precond_setup found about its spectrum bounds: read with the next scalars the host waits for.
chns_status pc_flags_fetch(Ctx& c) {
    CHNS_CUDA(cudaMemcpyAsync(c.ws->hsc + MAXSC - 1, precond_flags(c.m), sizeof(unsigned int), cudaMemcpyDeviceToHost, c.s));
    return CHNS_OK;
}
chns_status pc_flags_check(const Ctx& c) {
    unsigned int f = 0;
    std::memcpy(&f, c.ws->hsc + MAXSC - 1, sizeof(f));
    if (f & 1u) { chns_set_error("pressure Schur spectrum bound is not finite"); return CHNS_ENAN; }
    if (f & 2u) { chns_set_error("Cahn-Hilliard block spectrum bound is not finite"); return CHNS_ENAN; }
    return CHNS_OK;
}

}  // namespace

extern "C" chns_status chns_newton_step(const chns_mesh* mc, const chns_params* p, const chns_solver_opts* o,
                                        const double* U_old, double* U, chns_stats* stats, void* stream) {
    if (chns_require_q1(mc, "chns_newton_step") != CHNS_OK) return CHNS_EINVAL;
    chns_mesh* m = const_cast<chns_mesh*>(mc);
    PhysConst pc;
    chns_status st = chns_check_params(mc, p, &pc);
    if (st != CHNS_OK) return st;
    if (!o || !U_old || !U) { chns_set_error("null argument"); return CHNS_EINVAL; }
    if ((st = chns_check_rows(mc, U_old, 8)) != CHNS_OK || (st = chns_check_rows(mc, U, 8)) != CHNS_OK) return st;
    if (o->restart < 1 || o->restart > MAXSC / 4 || o->max_krylov < 1 || o->max_newton < 0 ||
        (o->precision != 0 && o->precision != 1) || (o->pc_type < 0 || o->pc_type > 4) ||
        (o->pc_type >= 1 && (o->pc_degree < 2 || o->pc_degree > 200)) ||
        !(o->ew_eta0 == 0.0 || (o->ew_eta0 > 0.0 && o->ew_eta0 < 1.0)) || (o->guess != 0 && o->guess != 1)) {
        chns_set_error("bad solver options (restart in [1, 256], max_krylov >= 1, precision 0/1, pc_type 0..4, "
                       "pc_degree in [2, 200], ew_eta0 0 or in (0, 1), guess 0/1)");
        return CHNS_EINVAL;
    }
    if ((st = ensure_ws(m, o->restart)) != CHNS_OK) return st;
    SolverWS* ws = m->ws;
    Ctx c{m, ws, (cudaStream_t)stream, ws->n, 0};
    c.g = grid_for(c.n);
    const int D = m->dm.dim, NF = m->dm.nf, mres = o->restart;
    const bool mixed = o->precision == 1;
    const int schur = o->pc_type >= 1 ? 1 : 0;
    const int chblk = (o->pc_type == 2 || o->pc_type == 4) ? 1 : 0;
    const bool use_mg = o->pc_type >= 3;   // pressure Schur by a multigrid V-cycle
    const int pcmask = schur | (chblk << 1);
    const int gN1 = (int)((m->dm.N + 255) / 256);
    PrecondSpec spec;
    spec.schur = schur;
    spec.mg = use_mg;
    spec.ch = chblk;
    spec.degree = o->pc_degree;
    if (chblk) {
        // Cahn-Hilliard block: S_phi ~ (1/dt)(M + eps K) M^{-1} (M + eps K), eps^2 = dt Cn/(2 Pe)
        spec.dt = (float)p->dt;
        spec.inv_pecn = (float)(1.0 / (p->Pe * p->Cn));
        spec.cn2 = (float)(p->Cn * p->Cn);
        spec.eps = (float)std::sqrt(p->dt * p->Cn / (2.0 * p->Pe));
    }
    if (schur && (st = precond_prepare(m, spec, c.s)) != CHNS_OK) return st;
    const int pin = p->pin_pressure;
    const int gN = (int)((m->dm.N + 127) / 128);
    chns_stats S;
    std::memset(&S, 0, sizeof(S));
    S.reason = CHNS_OK;

    CHNS_CUDA(cudaMemsetAsync(m->d_flags, 0, sizeof(unsigned int), c.s));
    if (o->guess == 0) { copy64_kernel<<<c.g, 256, 0, c.s>>>(U_old, U, c.n); chns_count_launches(1); }
    if (mixed) { to32_kernel<<<c.g, 256, 0, c.s>>>(U_old, ws->Uo32, c.n); chns_count_launches(1); }
    CHNS_CUDA(cudaGetLastError());

    std::vector<double> H((size_t)(mres + 1) * mres), cs(mres), sn(mres), gv(mres + 1), y(mres);
    double r0 = 0.0, rn = 0.0;
    chns_status result = CHNS_OK;
    // m_p^T z of the pin-mode-2 operator J + u m_p^T / |Omega|: formed with the pressure rows of z by
    // the pressure preconditioner, or by a pass of its own
    PrecondMean pmn;
    if (pin == 2) {
        pmn.nmass = m->d_nmass;
        pmn.partials = ws->mpart;
        pmn.counter = ws->counter + krylov::COUNTERS;
        pmn.out = ws->sc + SC_MEAN;
    }
    // Gram-Schmidt of Arnoldi step j on w = S J z (+ the rank-one term), with device-decided
    // re-orthogonalisation, and the read-back of the Hessenberg column
    const double thr = 0.01;
    auto orth_enqueue = [&](cudaStream_t st, int j) -> int {
        const double* mean = pin == 2 ? ws->sc + SC_MEAN : nullptr;
        const krylov::Source src{mixed ? ws->y32 : nullptr, mixed ? nullptr : ws->t64, ws->S, mean, 1.0 / m->volume, NF, D};
        return krylov::orthogonalise(ws->V, ws->ld, j + 1, src, c.n, ws->sc, thr, ws->hsc, ws->part, ws->counter, st);
    };
    auto build_pc = [&]() -> chns_status {
        CHNS_CUDA(cudaEventRecord(ws->ev[2], c.s));
        if (mixed) {
            { to32_kernel<<<c.g, 256, 0, c.s>>>(U, ws->Us32, c.n); chns_count_launches(1); }
            CHNS_CUDA(launch_pc_build(m, pc, ws->Uo32, ws->Us32, ws->Pblk32, ws->ce, c.s));
            { pc_invert_kernel<float, float><<<gN, 128, 0, c.s>>>(m->dm, ws->Pblk32, ws->Pinv32, pin, ws->S, ws->Sd, pcmask); chns_count_launches(1); }
        } else {
            CHNS_CUDA(launch_pc_build(m, pc, U_old, U, ws->Pblk64, ws->ce, c.s));
            { pc_invert_kernel<double, double><<<gN, 128, 0, c.s>>>(m->dm, ws->Pblk64, ws->Pinv64, pin, ws->S, ws->Sd, pcmask); chns_count_launches(1); }
        }
        CHNS_CUDA(cudaGetLastError());
        if (chblk) {
            if (mixed) ch_nodal_kernel<float><<<gN1, 256, 0, c.s>>>(m->dm.N, NF, D + 1, ws->Uo32, ws->Us32, ws->ch_psi2);
            else ch_nodal_kernel<double><<<gN1, 256, 0, c.s>>>(m->dm.N, NF, D + 1, U_old, U, ws->ch_psi2);
            chns_count_launches(1);
        }
        if (schur) {
            chns_status st3 = precond_setup(m, spec, ws->ce, ws->ch_psi2, c.s);
            if (st3 == CHNS_OK) st3 = pc_flags_fetch(c);
            if (st3 != CHNS_OK) return st3;
        }
        CHNS_CUDA(cudaEventRecord(ws->ev[3], c.s));
        return CHNS_OK;
    };
    // m_p^T v of vectors that do not come from the pressure preconditioner
    const double inv_vol = 1.0 / m->volume;
    const int nbm = c.g < 1024 ? c.g : 1024;
    auto pmean = [&](const auto* v) {
        { field_mass_kernel<<<nbm, 256, 0, c.s>>>(m->d_nmass, v, NF, D, m->dm.N, m->d_partials); chns_count_launches(1); }
        { final_reduce_kernel<<<1, 256, 0, c.s>>>(m->d_partials, nbm, 1, ws->sc + SC_MEAN); chns_count_launches(1); }
    };
    bool pc_pending = false;
    double eta_prev = 0.0, rn_prev = 0.0;   // previous forcing term and residual (Eisenstat-Walker)
    for (int it = 0;; ++it) {
        CHNS_CUDA(launch_residual(m, pc, U_old, U, ws->R, pin, c.s));
        if (it == 0) {
            // row equilibration of the step (1/|diag J| at U^0): the Newton test and the
            // Krylov residual weigh every field by its own scale (the pressure rows carry
            // coefficients ~ tau/We and would otherwise be invisible in ||R||)
            if ((st = build_pc()) != CHNS_OK) return st;
            pc_pending = true;
            { copy64_kernel<<<c.g, 256, 0, c.s>>>(ws->S, ws->S0, c.n); chns_count_launches(1); }
        }
        { scale_vec_kernel<double><<<c.g, 256, 0, c.s>>>(ws->R, ws->S0, ws->SR, 1.0, c.n); chns_count_launches(1); }
        if ((st = dot_host(c, ws->SR, ws->SR, &rn)) != CHNS_OK) return st;
        if (schur && (st = pc_flags_check(c)) != CHNS_OK) return st;
        unsigned int flag = 0;
        CHNS_CUDA(cudaMemcpy(&flag, m->d_flags, sizeof(unsigned int), cudaMemcpyDeviceToHost));
        rn = std::sqrt(rn);
        if (it == 0) r0 = rn;
        S.newton_its = it;
        if (it < CHNS_HIST) S.res_hist[it] = rn;
        S.res0 = r0;
        S.res_final = rn;
        if (flag & 1u) { chns_set_error("a tau_m radicand was not positive"); result = CHNS_ETAU; break; }
        if (!std::isfinite(rn)) { chns_set_error("non-finite residual norm"); result = CHNS_ENAN; break; }
        if (rn <= o->atol || rn <= o->rtol * r0) break;
        if (it >= o->max_newton) { chns_set_error("Newton did not converge"); result = CHNS_ENOCONV; break; }

        // linearisation state and preconditioner (already built for the first iterate)
        if (it > 0) {
            if ((st = build_pc()) != CHNS_OK) return st;
            pc_pending = true;
        }

        // GMRES(mres) on J dU = -R, right preconditioned, from dU = 0
        CHNS_CUDA(cudaMemsetAsync(ws->dU, 0, c.n * sizeof(double), c.s));
        double rnorm = rn;
        int kry = 0;
        // r = -S R (S: row equilibration of this linearisation), in slot 0 of the basis
        { scale_vec_kernel<double><<<c.g, 256, 0, c.s>>>(ws->R, ws->S, ws->V, -1.0, c.n); chns_count_launches(1); }
        {
            double bb;
            if ((st = dot_host(c, ws->V, ws->V, &bb)) != CHNS_OK) return st;
            if (schur && (st = pc_flags_check(c)) != CHNS_OK) return st;
            rnorm = std::sqrt(bb);
        }
        const double bnorm_s = rnorm;
        // forcing term: krylov_rtol (or the Eisenstat-Walker term with ew_eta0 > 0),
        // relaxed once the Newton target is near (a solve below a tenth of what the
        // target needs is wasted)
        const double target = std::max(o->atol, o->rtol * r0);
        double eta_k = o->krylov_rtol;
        if (o->ew_eta0 > 0.0) {
            // Eisenstat-Walker choice 2 (gamma 0.9, alpha 2) with their safeguard
            if (it == 0) {
                eta_k = o->ew_eta0;
            } else {
                const double ratio = rn / rn_prev;
                eta_k = 0.9 * ratio * ratio;
                const double guard = 0.9 * eta_prev * eta_prev;
                if (guard > 0.1) eta_k = std::max(eta_k, guard);
            }
            eta_k = std::min(0.9, std::max(o->krylov_rtol, eta_k));
        }
        const double eta = std::max(eta_k, std::min(0.5, 0.1 * target / rn));
        eta_prev = eta_k;
        rn_prev = rn;
        // z = M^{-1} S^{-1} v_j and y = J z; w = S y (similarity scaling: the eigenvalues of S J M^{-1}
        // S^{-1} are those of J M^{-1}) is formed by the dot pass that reads it.  The J x / apply
        // timing events come from set es (two sets alternate, so the next vector's application can
        // be queued before this one's events are read)
        auto apply_op = [&](int j, int es) -> chns_status {
            const double *Vj = ws->V + (size_t)j * ws->ld, *sj = ws->sc + SC_SCALE + j;
            cudaEvent_t* E = ws->ev + 8 * es;
            if (j == 0) CHNS_CUDA(cudaEventRecord(E[4], c.s));   // later ones start where the Gram-Schmidt pass ended
            if (mixed) {
                launch_pc_first<false>(m, pcmask, ws->Pinv32, Vj, sj, ws->Sd, ws->z32, c.s);
                if (schur && (st = precond_apply(m, spec, ws->z32, pmn, c.s)) != CHNS_OK) return st;
                if (pin == 2 && !schur) pmean(ws->z32);
                CHNS_CUDA(cudaEventRecord(E[5], c.s));
                CHNS_CUDA(launch_jvp32(m, pc, ws->Uo32, ws->Us32, ws->z32, ws->y32, pin, c.s));
            } else {
                launch_pc_first<false>(m, pcmask, ws->Pinv64, Vj, sj, ws->Sd, ws->z64, c.s);
                if (schur && (st = precond_apply(m, spec, ws->z64, pmn, c.s)) != CHNS_OK) return st;
                if (pin == 2 && !schur) pmean(ws->z64);
                CHNS_CUDA(cudaEventRecord(E[5], c.s));
                CHNS_CUDA(launch_jvp64(m, pc, U_old, U, ws->z64, ws->t64, pin, c.s));
            }
            CHNS_CUDA(cudaEventRecord(E[1], c.s));
            CHNS_CUDA(cudaGetLastError());
            S.jvp_calls++;
            return CHNS_OK;
        };
        while (true) {
            // v_0 = r / ||r||: r is in slot 0
            double beta = rnorm;
            { set_scalar_kernel<<<1, 1, 0, c.s>>>(ws->sc + SC_SCALE, 1.0 / beta); chns_count_launches(1); }
            std::fill(gv.begin(), gv.end(), 0.0);
            gv[0] = beta;
            int j = 0;
            bool done = false;
            if ((st = apply_op(0, 0)) != CHNS_OK) return st;
            for (; j < mres && kry < o->max_krylov; ++j, ++kry) {
                const int es = j & 1;
                // classical Gram-Schmidt with selective re-orthogonalisation (decided on the
                // device) and the next Arnoldi vector, all queued without a host round trip
                cudaEvent_t* E = ws->ev + 8 * es;
                chns_count_launches(orth_enqueue(c.s, j));
                CHNS_CUDA(cudaGetLastError());
                CHNS_CUDA(cudaEventRecord(E[7], c.s));
                // queue the next vector's operator application before reading the scalars, so
                // the GPU works on it while the host updates the Hessenberg column; if this
                // iteration turns out to be the last one, that result is simply not used
                if (j + 1 < mres && kry + 1 < o->max_krylov)
                    if ((st = apply_op(j + 1, es ^ 1)) != CHNS_OK) return st;
                CHNS_CUDA(cudaEventSynchronize(E[7]));
                {
                    float ms = 0.0f;
                    CHNS_CUDA(cudaEventElapsedTime(&ms, E[5], E[1]));
                    S.jvp_ms += ms;
                    CHNS_CUDA(cudaEventElapsedTime(&ms, j == 0 ? E[4] : ws->ev[8 * (es ^ 1) + 7], E[5]));
                    S.apply_ms += ms;
                    CHNS_CUDA(cudaEventElapsedTime(&ms, E[1], E[7]));
                    S.orth_ms += ms;
                    if (pc_pending) {
                        CHNS_CUDA(cudaEventElapsedTime(&ms, ws->ev[2], ws->ev[3]));
                        S.pc_ms += ms;
                        pc_pending = false;
                    }
                }
                const double hn = std::sqrt(ws->hsc[SC_NA]);
                for (int i = 0; i <= j; ++i) H[(size_t)i * mres + j] = ws->hsc[i];
                H[(size_t)(j + 1) * mres + j] = hn;
                if (!std::isfinite(hn)) { chns_set_error("non-finite Arnoldi vector"); S.reason = CHNS_EBREAKDOWN; result = CHNS_EBREAKDOWN; break; }
                // Givens rotations
                for (int i = 0; i < j; ++i) {
                    const double a = H[(size_t)i * mres + j], b = H[(size_t)(i + 1) * mres + j];
                    H[(size_t)i * mres + j] = cs[i] * a + sn[i] * b;
                    H[(size_t)(i + 1) * mres + j] = -sn[i] * a + cs[i] * b;
                }
                const double a = H[(size_t)j * mres + j], b = H[(size_t)(j + 1) * mres + j];
                const double r = std::hypot(a, b);
                cs[j] = r > 0 ? a / r : 1.0;
                sn[j] = r > 0 ? b / r : 0.0;
                H[(size_t)j * mres + j] = r;
                H[(size_t)(j + 1) * mres + j] = 0.0;
                gv[j + 1] = -sn[j] * gv[j];
                gv[j] = cs[j] * gv[j];
                rnorm = std::fabs(gv[j + 1]);
                if (rnorm <= eta * bnorm_s || hn == 0.0) {
                    ++j;
                    ++kry;
                    done = true;
                    break;
                }
            }
            if (result != CHNS_OK) break;
            // y = H^{-1} g, dU += M^{-1} V y
            const int k = j;
            for (int i = k - 1; i >= 0; --i) {
                double s = gv[i];
                for (int l = i + 1; l < k; ++l) s -= H[(size_t)i * mres + l] * y[l];
                y[i] = s / H[(size_t)i * mres + i];
            }
            std::memcpy(ws->hsc, y.data(), k * sizeof(double));
            CHNS_CUDA(cudaMemcpyAsync(ws->sc, ws->hsc, k * sizeof(double), cudaMemcpyHostToDevice, c.s));
            krylov::combine(ws->V, ws->ld, k, ws->sc, ws->sc + SC_SCALE, ws->SR, c.n, c.s);
            chns_count_launches(1);
            if (mixed) launch_pc_first<false>(m, pcmask, ws->Pinv32, ws->SR, nullptr, ws->Sd, ws->z64, c.s);
            else launch_pc_first<false>(m, pcmask, ws->Pinv64, ws->SR, nullptr, ws->Sd, ws->z64, c.s);
            if (schur && (st = precond_apply(m, spec, ws->z64, PrecondMean(), c.s)) != CHNS_OK) return st;
            { axpy_kernel<<<c.g, 256, 0, c.s>>>(1.0, ws->z64, ws->dU, c.n); chns_count_launches(1); }
            CHNS_CUDA(cudaGetLastError());
            if (done || kry >= o->max_krylov) break;
            // restart: r = -R - J dU (same operator as the Arnoldi process)
            if (mixed) {
                { to32_kernel<<<c.g, 256, 0, c.s>>>(ws->dU, ws->z32, c.n); chns_count_launches(1); }
                CHNS_CUDA(cudaEventRecord(ws->ev[0], c.s));
                CHNS_CUDA(launch_jvp32(m, pc, ws->Uo32, ws->Us32, ws->z32, ws->y32, pin, c.s));
                CHNS_CUDA(cudaEventRecord(ws->ev[1], c.s));
                { to64_kernel<<<c.g, 256, 0, c.s>>>(ws->y32, ws->w, c.n); chns_count_launches(1); }
            } else {
                CHNS_CUDA(cudaEventRecord(ws->ev[0], c.s));
                CHNS_CUDA(launch_jvp64(m, pc, U_old, U, ws->dU, ws->w, pin, c.s));
                CHNS_CUDA(cudaEventRecord(ws->ev[1], c.s));
            }
            S.jvp_calls++;
            { axpby_kernel<<<c.g, 256, 0, c.s>>>(-1.0, ws->R, -1.0, ws->w, c.n); chns_count_launches(1); }
            if (pin == 2) {
                pmean(ws->dU);
                { scale_vec_pmean_kernel<double><<<c.g, 256, 0, c.s>>>(ws->w, ws->S, ws->V, c.n, NF, D, ws->sc + SC_MEAN, -inv_vol); chns_count_launches(1); }
            } else {
                { scale_vec_kernel<double><<<c.g, 256, 0, c.s>>>(ws->w, ws->S, ws->V, 1.0, c.n); chns_count_launches(1); }
            }
            double rr;
            if ((st = dot_host(c, ws->V, ws->V, &rr)) != CHNS_OK) return st;
            rnorm = std::sqrt(rr);
            {
                float ms = 0.0f;
                CHNS_CUDA(cudaEventElapsedTime(&ms, ws->ev[0], ws->ev[1]));
                S.jvp_ms += ms;
            }
            if (rnorm <= eta * bnorm_s) break;
        }
        S.krylov_its += kry;
        if (it < CHNS_HIST) S.krylov_hist[it] = kry;
        if (result != CHNS_OK) break;
        if (pin == 2) {
            // keep int p^{k+1} = int p^k: remove the mean of the pressure update (the
            // constant pressure spans the null space of J when no row is pinned)
            const int nbk = c.g < 1024 ? c.g : 1024;
            { field_mass_kernel<<<nbk, 256, 0, c.s>>>(m->d_nmass, ws->dU, NF, D, m->dm.N, m->d_partials); chns_count_launches(1); }
            { final_reduce_kernel<<<1, 256, 0, c.s>>>(m->d_partials, nbk, 1, ws->sc + 600); chns_count_launches(1); }
            { field_shift_kernel<<<c.g, 256, 0, c.s>>>(ws->dU, NF, D, m->dm.N, ws->sc + 600, 1.0 / m->volume); chns_count_launches(1); }
            CHNS_CUDA(cudaGetLastError());
        }
        {
            // keep int phi^{k+1} = int phi^k (Proposition 1, exact for the solution of the
            // discrete system) for every inexact iterate too: shift the phi update by the
            // constant that removes the mass change (the nodal masses sum to |Omega|)
            const int nbk = c.g < 1024 ? c.g : 1024;
            { field_mass3_kernel<<<nbk, 256, 0, c.s>>>(m->d_nmass, U, ws->dU, U_old, NF, D + 1, m->dm.N, m->d_partials); chns_count_launches(1); }
            { final_reduce_kernel<<<1, 256, 0, c.s>>>(m->d_partials, nbk, 1, ws->sc + 606); chns_count_launches(1); }
            { field_shift_kernel<<<c.g, 256, 0, c.s>>>(ws->dU, NF, D + 1, m->dm.N, ws->sc + 606, 1.0 / m->volume); chns_count_launches(1); }
            CHNS_CUDA(cudaGetLastError());
        }
        { axpy_kernel<<<c.g, 256, 0, c.s>>>(1.0, ws->dU, U, c.n); chns_count_launches(1); }
        double du;
        if ((st = dot_host(c, ws->dU, ws->dU, &du)) != CHNS_OK) return st;
        S.du_norm = std::sqrt(du);
    }
    // a breakdown leaves the next vector's operator application in flight, on the caller's vectors and on
    // the preconditioner's device description, which the next call may rewrite
    if (result == CHNS_EBREAKDOWN) CHNS_CUDA(cudaStreamSynchronize(c.s));
    S.reason = result;
    if (stats) *stats = S;
    return result;
}

// ---------------------------------------------------------------------------------
// Adjoint of one implicit step (reverse mode through Section 3.4's solve): with
// R(U^k, U^{k+1}; Cn) = 0, a cotangent g of U^{k+1} gives J^T lambda = P^T g
// (J = dR/dU^{k+1}; P the pressure-level normalisation of pin mode 2) and the
// cotangents -(dR/dU^k)^T lambda of U^k and -(dR/dCn)^T lambda of Cn.
// ---------------------------------------------------------------------------------
namespace {

// unweighted sum of field f into per-block partials
__global__ void field_sum_kernel(const double* __restrict__ v, int NF, int f, int64_t N, double* partials) {
    double acc[1] = {0.0};
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x)
        acc[0] += v[(size_t)n * NF + f];
    block_reduce_store<1>(acc, partials);
}
// out = sum_n wt[n*NF + f] v[n*NF + f]: the block that finishes last sums the partials
__global__ void field_wdot_kernel(const double* __restrict__ wt, const double* __restrict__ v, int NF, int f,
                                  int64_t N, double* partials, unsigned int* counter, double* out) {
    double acc[1] = {0.0};
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x)
        acc[0] += wt[(size_t)n * NF + f] * v[(size_t)n * NF + f];
    block_reduce_store<1>(acc, partials);
    if (!krylov::last_block(counter) || threadIdx.x >= 32) return;
    double t = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) t += __ldcg(partials + b);
    t = krylov::warp_sum(t);
    if (threadIdx.x == 0) out[0] = t;
}
// v[n*NF + f] += a * m[n] * sc[0]
__global__ void field_axpy_mass_kernel(double* __restrict__ v, int NF, int f, int64_t N, const double* __restrict__ m,
                                       const double* __restrict__ sc, double a) {
    const double s = a * sc[0];
    for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < N; n += (int64_t)gridDim.x * blockDim.x)
        v[(size_t)n * NF + f] += s * m[n];
}

}  // namespace

extern "C" chns_status chns_step_adjoint(const chns_mesh* mc, const chns_params* p, const chns_solver_opts* o,
                                         const double* U_old, const double* U_new, const double* g, double* lambda,
                                         double* gU_old, double* gCn, chns_stats* stats, void* stream) {
    if (chns_require_q1(mc, "chns_step_adjoint") != CHNS_OK) return CHNS_EINVAL;
    chns_mesh* m = const_cast<chns_mesh*>(mc);
    PhysConst pc;
    chns_status st = chns_check_params(mc, p, &pc);
    if (st != CHNS_OK) return st;
    if (!o || !U_old || !U_new || !g || !lambda || !gU_old) { chns_set_error("null argument"); return CHNS_EINVAL; }
    if ((st = chns_check_rows(mc, U_old, 8)) != CHNS_OK || (st = chns_check_rows(mc, U_new, 8)) != CHNS_OK) return st;
    if (o->restart < 1 || o->restart > MAXSC / 4 || o->max_krylov < 1 || o->pc_type < 0 || o->pc_type > 4 ||
        (o->pc_type >= 1 && (o->pc_degree < 2 || o->pc_degree > 200))) {
        chns_set_error("bad solver options (restart in [1, 256], max_krylov >= 1, pc_type 0..4, pc_degree in [2, 200])");
        return CHNS_EINVAL;
    }
    if ((st = ensure_ws(m, o->restart)) != CHNS_OK) return st;
    SolverWS* ws = m->ws;
    Ctx c{m, ws, (cudaStream_t)stream, ws->n, 0};
    c.g = grid_for(c.n);
    const int D = m->dm.dim, NF = m->dm.nf, mres = o->restart, pin = p->pin_pressure;
    // the pressure Schur approximation is symmetric, so J^T takes it as J does; the
    // Cahn-Hilliard block of pc_type 2 / 4 is not used here
    const bool schur = o->pc_type >= 1;
    PrecondSpec spec;
    spec.schur = schur;
    spec.mg = o->pc_type >= 3;
    spec.degree = o->pc_degree;
    if (schur && (st = precond_prepare(m, spec, c.s)) != CHNS_OK) return st;
    const int gN = (int)((m->dm.N + 127) / 128);
    const int nbk = c.g < 1024 ? c.g : 1024;
    const int nbw = std::min(grid_for(m->dm.N), 512);
    chns_stats S;
    std::memset(&S, 0, sizeof(S));

    // nodal blocks of J (FP64) at the converged state; J^T's blocks are their transposes
    CHNS_CUDA(launch_pc_build(m, pc, U_old, U_new, ws->Pblk64, ws->ce, c.s));
    { pc_invert_kernel<double, double><<<gN, 128, 0, c.s>>>(m->dm, ws->Pblk64, ws->Pinv64, pin, ws->S, ws->Sd, schur ? 1 : 0); chns_count_launches(1); }
    if (schur) {
        if ((st = precond_setup(m, spec, ws->ce, nullptr, c.s)) != CHNS_OK) return st;
        if ((st = pc_flags_fetch(c)) != CHNS_OK) return st;
    }
    // pin mode 2: J' = J + u m_p^T / |Omega| with u = |diag J| on the pressure rows is
    // nonsingular, and J'^T lambda = P^T g has the solution of J^T lambda = P^T g with
    // u^T lambda = 0 (GMRES on the singular J^T drifts along its null vector)
    const double inv_vol = 1.0 / m->volume;
    auto add_pmean_T = [&](const double* v, double* y) {
        { field_wdot_kernel<<<nbw, 256, 0, c.s>>>(ws->Sd, v, NF, D, m->dm.N, m->d_partials, ws->counter + krylov::COUNTERS, ws->sc + SC_MISC + 1); chns_count_launches(1); }
        { field_axpy_mass_kernel<<<c.g, 256, 0, c.s>>>(y, NF, D, m->dm.N, m->d_nmass, ws->sc + SC_MISC + 1, inv_vol); chns_count_launches(1); }
    };
    // b = P^T g: remove sum(g_p) * m / |Omega| from the pressure part (pin mode 2)
    double* b = ws->R;
    { copy64_kernel<<<c.g, 256, 0, c.s>>>(g, b, c.n); chns_count_launches(1); }
    if (pin == 2) {
        { field_sum_kernel<<<nbk, 256, 0, c.s>>>(g, NF, D, m->dm.N, m->d_partials); chns_count_launches(1); }
        { final_reduce_kernel<<<1, 256, 0, c.s>>>(m->d_partials, nbk, 1, ws->sc + SC_MISC); chns_count_launches(1); }
        { field_axpy_mass_kernel<<<c.g, 256, 0, c.s>>>(b, NF, D, m->dm.N, m->d_nmass, ws->sc + SC_MISC, -1.0 / m->volume); chns_count_launches(1); }
    }
    CHNS_CUDA(cudaGetLastError());
    double bb;
    if ((st = dot_host(c, b, b, &bb)) != CHNS_OK) return st;
    if (schur && (st = pc_flags_check(c)) != CHNS_OK) return st;
    const double bnorm = std::sqrt(bb);
    CHNS_CUDA(cudaMemsetAsync(lambda, 0, c.n * sizeof(double), c.s));
    S.res0 = bnorm;
    chns_status result = CHNS_OK;
    if (bnorm > 0.0) {
        // right-preconditioned GMRES on J^T M^{-T} y = b, lambda = M^{-T} y
        std::vector<double> H((size_t)(mres + 1) * mres), cs(mres), sn(mres), gv(mres + 1), y(mres);
        double rnorm = bnorm;
        int kry = 0;
        { copy64_kernel<<<c.g, 256, 0, c.s>>>(b, ws->V, c.n); chns_count_launches(1); }
        // slot j + 1 = J^T M^{-T} v_j
        auto apply_op = [&](int j) -> chns_status {
            double* w = ws->V + (size_t)(j + 1) * ws->ld;
            launch_pc_first<true>(m, schur ? 1 : 0, ws->Pinv64, ws->V + (size_t)j * ws->ld, ws->sc + SC_SCALE + j, nullptr, ws->z64, c.s);
            if (schur && (st = precond_apply(m, spec, ws->z64, PrecondMean(), c.s)) != CHNS_OK) return st;
            CHNS_CUDA(launch_vjp(m, pc, U_old, U_new, ws->z64, w, nullptr, nullptr, pin, c.s));
            if (pin == 2) add_pmean_T(ws->z64, w);
            S.jvp_calls++;
            return CHNS_OK;
        };
        while (true) {
            const double beta = rnorm;
            { set_scalar_kernel<<<1, 1, 0, c.s>>>(ws->sc + SC_SCALE, 1.0 / beta); chns_count_launches(1); }
            std::fill(gv.begin(), gv.end(), 0.0);
            gv[0] = beta;
            int j = 0;
            bool done = false;
            if ((st = apply_op(0)) != CHNS_OK) return st;
            for (; j < mres && kry < o->max_krylov; ++j, ++kry) {
                // two full Gram-Schmidt passes, then the next vector's operator queued
                // before the host waits for this one's column
                const krylov::Source src{nullptr, nullptr, nullptr, nullptr, 0.0, NF, D};
                chns_count_launches(krylov::orthogonalise(ws->V, ws->ld, j + 1, src, c.n, ws->sc, HUGE_VAL, ws->hsc, ws->part, ws->counter, c.s));
                CHNS_CUDA(cudaGetLastError());
                CHNS_CUDA(cudaEventRecord(ws->ev[10], c.s));
                if (j + 1 < mres && kry + 1 < o->max_krylov)
                    if ((st = apply_op(j + 1)) != CHNS_OK) return st;
                CHNS_CUDA(cudaEventSynchronize(ws->ev[10]));
                const double hn = std::sqrt(ws->hsc[SC_NA]);
                for (int i = 0; i <= j; ++i) H[(size_t)i * mres + j] = ws->hsc[i];
                H[(size_t)(j + 1) * mres + j] = hn;
                if (!std::isfinite(hn)) { chns_set_error("non-finite Arnoldi vector"); result = CHNS_EBREAKDOWN; break; }
                for (int i = 0; i < j; ++i) {
                    const double a = H[(size_t)i * mres + j], bq = H[(size_t)(i + 1) * mres + j];
                    H[(size_t)i * mres + j] = cs[i] * a + sn[i] * bq;
                    H[(size_t)(i + 1) * mres + j] = -sn[i] * a + cs[i] * bq;
                }
                const double a = H[(size_t)j * mres + j], bq = H[(size_t)(j + 1) * mres + j];
                const double r = std::hypot(a, bq);
                cs[j] = r > 0 ? a / r : 1.0;
                sn[j] = r > 0 ? bq / r : 0.0;
                H[(size_t)j * mres + j] = r;
                H[(size_t)(j + 1) * mres + j] = 0.0;
                gv[j + 1] = -sn[j] * gv[j];
                gv[j] = cs[j] * gv[j];
                rnorm = std::fabs(gv[j + 1]);
                if (rnorm <= o->krylov_rtol * bnorm || hn == 0.0) {
                    ++j;
                    ++kry;
                    done = true;
                    break;
                }
            }
            if (result != CHNS_OK) break;
            const int k = j;
            for (int i = k - 1; i >= 0; --i) {
                double sacc = gv[i];
                for (int l = i + 1; l < k; ++l) sacc -= H[(size_t)i * mres + l] * y[l];
                y[i] = sacc / H[(size_t)i * mres + i];
            }
            std::memcpy(ws->hsc, y.data(), k * sizeof(double));
            CHNS_CUDA(cudaMemcpyAsync(ws->sc, ws->hsc, k * sizeof(double), cudaMemcpyHostToDevice, c.s));
            krylov::combine(ws->V, ws->ld, k, ws->sc, ws->sc + SC_SCALE, ws->t64, c.n, c.s);
            chns_count_launches(1);
            launch_pc_first<true>(m, schur ? 1 : 0, ws->Pinv64, ws->t64, nullptr, nullptr, ws->z64, c.s);
            if (schur && (st = precond_apply(m, spec, ws->z64, PrecondMean(), c.s)) != CHNS_OK) return st;
            { axpy_kernel<<<c.g, 256, 0, c.s>>>(1.0, ws->z64, lambda, c.n); chns_count_launches(1); }
            CHNS_CUDA(cudaGetLastError());
            if (done || kry >= o->max_krylov) break;
            // restart: r = b - J^T lambda
            CHNS_CUDA(launch_vjp(m, pc, U_old, U_new, lambda, ws->V, nullptr, nullptr, pin, c.s));
            if (pin == 2) add_pmean_T(lambda, ws->V);
            S.jvp_calls++;
            { axpby_kernel<<<c.g, 256, 0, c.s>>>(1.0, b, -1.0, ws->V, c.n); chns_count_launches(1); }
            double rr;
            if ((st = dot_host(c, ws->V, ws->V, &rr)) != CHNS_OK) return st;
            rnorm = std::sqrt(rr);
            if (rnorm <= o->krylov_rtol * bnorm) break;
        }
        S.krylov_its = kry;
        S.res_final = rnorm;
        if (result == CHNS_OK && rnorm > o->krylov_rtol * bnorm * 1.0001) {
            chns_set_error("adjoint GMRES did not reach krylov_rtol within max_krylov");
            result = CHNS_ENOCONV;
        }
    }
    // cotangents of U^k and Cn: -(dR/dU^k)^T lambda, -(dR/dCn)^T lambda
    CHNS_CUDA(launch_vjp(m, pc, U_old, U_new, lambda, ws->t64, gU_old, gCn, pin, c.s));
    { axpby_kernel<<<c.g, 256, 0, c.s>>>(0.0, gU_old, -1.0, gU_old, c.n); chns_count_launches(1); }
    if (gCn) { axpby_kernel<<<1, 32, 0, c.s>>>(0.0, gCn, -1.0, gCn, 1); chns_count_launches(1); }
    if (pin == 2) {
        // the normalisation int p^{k+1} = int p^k passes sum(g_p) m / |Omega| to p^k
        { field_axpy_mass_kernel<<<c.g, 256, 0, c.s>>>(gU_old, NF, D, m->dm.N, m->d_nmass, ws->sc + SC_MISC, 1.0 / m->volume); chns_count_launches(1); }
    }
    CHNS_CUDA(cudaGetLastError());
    CHNS_CUDA(cudaStreamSynchronize(c.s));
    S.reason = result;
    if (stats) *stats = S;
    return result;
}
