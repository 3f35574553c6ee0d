// Programmatic dependent launch: a kernel launched as a link may start while its predecessor on the
// stream runs (from when all of that one's blocks called chain_next, or at its end), and must call
// chain_wait, in every thread, before it touches what an earlier kernel of the chain writes.
#pragma once

#include <cuda_runtime.h>

template <bool ON> __device__ __forceinline__ void chain_next() {
    if (ON) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <bool ON> __device__ __forceinline__ void chain_wait() {
    if (ON) asm volatile("griddepcontrol.wait;" ::: "memory");
}
// LINKED: as a link; else an ordinary launch
template <bool LINKED, class... P, class... A>
cudaError_t chain(void (*kernel)(P...), unsigned grid, int threads, cudaStream_t st, A... args) {
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cfg.attrs = &a;
    cfg.numAttrs = LINKED ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);   // also left for cudaGetLastError
}
