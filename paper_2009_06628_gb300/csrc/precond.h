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
// Overwrites the pressure (schur) and phi, mu (ch) rows of z with the preconditioned rows of the
// FP64 vector v.  Replayed from a CUDA graph per (v, z, spec).
chns_status precond_apply(chns_mesh* m, const PrecondSpec& spec, const double* v, float* z, cudaStream_t s);
chns_status precond_apply(chns_mesh* m, const PrecondSpec& spec, const double* v, double* z, cudaStream_t s);
// Captured graphs hold the callers' vectors: drop them when those are freed.
void precond_drop_graphs(chns_mesh* m);
void precond_free(PrecondWS* p);
