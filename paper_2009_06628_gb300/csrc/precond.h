// Scalar-operator preconditioners of the Newton and adjoint solves: the pressure
// Schur-complement approximation (Chebyshev polynomial or multigrid V-cycle) and the
// Cahn-Hilliard block, on assembled Q1 operators (precond.cu).
#pragma once

#include <cuda_runtime.h>

#include "chns_internal.h"

struct PrecondWS;   // owned by the mesh (chns_mesh::pre)

struct PrecondSpec {
    bool schur = false;      // pressure Schur approximation
    bool mg = false;         // as a V-cycle instead of a Chebyshev polynomial
    bool ch = false;         // Cahn-Hilliard block on phi and mu
    int degree = 0;          // Chebyshev degree (polynomial / smoother)
    float dt = 0.0f, inv_pecn = 0.0f, cn2 = 0.0f, eps = 0.0f;   // Cahn-Hilliard block
    bool operator==(const PrecondSpec& o) const {
        return schur == o.schur && mg == o.mg && ch == o.ch && degree == o.degree && dt == o.dt &&
               inv_pecn == o.inv_pecn && cn2 == o.cn2 && eps == o.eps;
    }
};

// Allocate and build what `spec` needs and does not depend on the linearisation (once per mesh).
chns_status precond_prepare(chns_mesh* m, const PrecondSpec& spec, cudaStream_t s);
// Assemble for the element coefficients ce = dt/(2 rho We) and, with spec.ch, the nodal
// psi''(phi~) (device, FP32).  Asynchronous; a spectrum bound that is not finite sets the flag
// word below.
chns_status precond_setup(chns_mesh* m, const PrecondSpec& spec, const float* ce, const float* psi2, cudaStream_t s);
// device word, zeroed by precond_setup: bit 0 Schur bound, bit 1 Cahn-Hilliard bound not finite
const unsigned int* precond_flags(const chns_mesh* m);
// Compact inputs (FP32, one value per node) that the caller writes before every application: the
// pressure, phi and mu rows of the vector.  Overwritten by the application.
struct PrecondIn {
    float *p = nullptr, *phi = nullptr, *mu = nullptr;
};
PrecondIn precond_inputs(const chns_mesh* m);
// m_p^T z_p: formed with the pressure result (null out: not wanted)
struct PrecondMean {
    const double* nmass = nullptr;
    double* partials = nullptr;        // N / 64 + 64
    unsigned int* counter = nullptr;   // zero
    double* out = nullptr;
};
// Writes the pressure (schur) and phi, mu (ch) rows of z from the inputs.  Replayed from a CUDA
// graph per (z, mean, spec), four of which are kept; precond_prepare with another degree or kind of
// pressure approximation drops them (there is one description of the one-block levels per mesh).
chns_status precond_apply(chns_mesh* m, const PrecondSpec& spec, float* z, const PrecondMean& mean, cudaStream_t s);
chns_status precond_apply(chns_mesh* m, const PrecondSpec& spec, double* z, const PrecondMean& mean, cudaStream_t s);
// Captured graphs hold the callers' vectors: drop them when those are freed.
void precond_drop_graphs(chns_mesh* m);
void precond_free(PrecondWS* p);
