// lbm_async.cuh -- what the step and the adjoint kernels share: cp.async copies from global to
// shared memory, and launches that overlap the end of the launch before them.
#pragma once
#include <cuda_runtime.h>

namespace lbm {

// Chained launches. A step launched with `chained` follows another step or adjoint launch of the
// same call on the stream, or the call's graph replays, and may start before it has ended: its CTAs
// take the places that are free, load their first headers, records and words (which no launch
// of the chain writes) and wait in grid_wait() until the launch before has completed and its
// results are visible. Everything that a launch of the chain writes, or reads from one, comes
// after grid_wait(), which every CTA executes: so completion is transitive along the chain. A
// launch lets the next one start (grid_release) only after its own grid_wait(), so no more than
// two are on the GPU at once and the start of the third (which empties L1) comes after the first
// has ended; words that share a cache line between CTAs and change from launch to launch are read
// past L1 (__ldcg). The first launch of a call is never chained (the tables may have been written
// by the work before it). Without the attribute both instructions do nothing.
// Against unchained launches of the same kernels, a step: 32^3 channel FP16 4.2 -> 3.1 us, 48^3 pack
// FP32 4.8 -> 3.7, 96^3 pack FP32 14.7 -> 13.6, 128^3 pack FP64 61 -> 59; 256^3 packs 1 %.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st,
                                  bool chained, A... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8_sa(unsigned sa, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4_sa(unsigned sa, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

}  // namespace lbm
