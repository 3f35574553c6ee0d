// Nodal blocks of J for the block-Jacobi preconditioner (block_jacobi.cu).
#pragma once

#include <cuda_runtime.h>

#include "chns_internal.h"

// blk (N x n_f x n_f) = the nodal blocks at (Uo, Un); ce (E) = dt/(2 We) times the element mean of
// 1/rho.  The output type is that of the arithmetic.
cudaError_t launch_pc_build(const chns_mesh* m, const PhysConst& pc, const float* Uo, const float* Un, float* blk,
                            float* ce, cudaStream_t s);
cudaError_t launch_pc_build(const chns_mesh* m, const PhysConst& pc, const double* Uo, const double* Un, double* blk,
                            float* ce, cudaStream_t s);
