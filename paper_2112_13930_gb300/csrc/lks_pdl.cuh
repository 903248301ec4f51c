// lks_pdl.cuh -- a step kernel that follows another on its stream starts early (programmatic dependent
// launch): the launch is processed while the predecessor drains, and the kernel waits for it to
// finish, with everything it wrote visible, before it touches memory.  Kernels of a few microseconds gain
// most (us per step, before -> after): 128 x 128 FP64 duct 14.3 -> 11.2, 36 x 69 x 80 FP32 channel 18.5 ->
// 15.9, 152 x 439 FP32 in place 2.34 -> 2.12, 256 x 257 FP32 2.62 -> 2.45.
//
// No kernel triggers its successor before it exits (griddepcontrol.launch_dependents at the start was
// slower: blocks that wait take the SMs the running kernel left free and then share them, duct 27 us a
// step).  The fused row kernel and the two-node kernel of 16-bit storage with two buffers are launched plainly:
// they gained nothing and lost 1-2 % to the loads below.
//
// After the wait, loads are plain (coherent) ones: the read-only path is defined for data that nobody
// writes during the kernel's lifetime, which here begins while the predecessor still writes.
#pragma once
#include <cuda_runtime.h>

namespace lks {

__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launch `kernel`, which calls pdl_wait() before its first access, so that it may start early.
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st,
                              A... args) {
    cudaLaunchConfig_t lc = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.gridDim = grid;
    lc.blockDim = dim3(block);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kernel, static_cast<P>(args)...);
}

}  // namespace lks
