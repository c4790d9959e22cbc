// Programmatic dependent launch: a kernel started by pdl_launch may become resident while its
// predecessor on the stream drains; its pdl_wait() holds each thread until every earlier kernel has
// completed and its writes are visible.  What an earlier kernel writes is read after it and by plain
// loads or cp.async, never by __ldg: the read-only path promises data that does not change during the
// kernel, which here begins before its predecessor ends.  pdl_trigger() lets a successor started the same way in from
// the moment all of a kernel's blocks are resident.
// Used by the mixed stage kernel, whose set-up (tables, cleared operands, tensor memory) reads nothing
// an earlier kernel writes: P1, 48,000 elements, 16 steps 2.04 -> 1.95 ms; P1, 960 elements, 9 steps
// 205 -> 158 us together with the third context; P3, 1,572,864 elements, unchanged.  The CUDA-core
// kernels have no such set-up and ran slower with it (FP64 P1, 1,296 elements, 10 steps 542 -> 1,423 us;
// FP32 P2 2.51 -> 2.79 ms).
#pragma once

#include <cuda_runtime.h>

namespace dg {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Params, typename... Args>
inline cudaError_t pdl_launch(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

}  // namespace dg
