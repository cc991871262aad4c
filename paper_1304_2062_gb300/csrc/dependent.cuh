// Programmatic dependent launches between the passes of one stream: a kernel
// lets the next one start (dependent_launch) while its last blocks still run,
// and the next one sets up (tables, barriers: nothing the previous kernels write)
// before it waits for them (dependent_wait: every earlier kernel of the stream
// has completed and its writes are visible). Blocks that return without waiting
// are harmless: the kernel as a whole is not complete before its waiting blocks.
// After a library kernel, which never lets its successor start, such a launch
// is an ordinary one.
// A kernel launched so may start while what it is going to read is still being
// written: none of that is read-only data for its lifetime, and it must not be read
// through the non-coherent path (__ldg, const __restrict__ pointers), which may hold what
// an earlier kernel read there. Such loads are __ldcg. (With __ldg in the row pass one
// in some two hundred inpaints issued back to back had a stale row.)
#pragma once

#include <cuda_runtime.h>

namespace se2n {

__device__ __forceinline__ void dependent_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void dependent_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch fn so that it may start before the previous kernel of the stream has
// ended; fn must call dependent_wait before it touches what that one writes or reads.
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*fn)(P...), int grid, int block, size_t smem, cudaStream_t s, A... a) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, static_cast<P>(a)...);
}

}  // namespace se2n
