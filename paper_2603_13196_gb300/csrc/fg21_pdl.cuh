// Programmatic dependent launch for the likelihood's kernel chain (prep ->
// tensor or SIMT kernel -> reduction).  A kernel launched with
// launch_dependent() is scheduled as the blocks of the kernel before it in the
// stream exit, without the full kernel boundary in between, so its launch
// latency overlaps that kernel's tail (about 1 us per edge).  Every such
// kernel calls pdl_wait() before it reads or writes anything the earlier
// kernels touch: the wait returns once the preceding grid has completed and
// its memory operations are visible (and, through that grid's own wait,
// everything before it).  The wait is a no-op for a kernel launched the
// ordinary way.  No kernel triggers its dependents early: measured, the
// dependents' blocks then sit on the SMs beside the running kernel and cost
// more than the overlap gains.
//
// What the earlier kernels of the chain write must not be read before the wait.
// __restrict__ on a kernel's pointer and __ldg let the compiler move a load whose
// address it knows to before it, so:
//  - a kernel that reads a descriptor which the call's first kernel may have stored
//    has no __restrict__ on that parameter (a function called after the wait may);
//  - __ldg is for addresses that were themselves read after the wait, by a plain
//    load: not in a kernel whose descriptor is an argument by value.
// (As no kernel triggers its dependents early, every block that writes has ended
// when a reader's first block starts.)  With plain loads in the tensor kernel
// instead of __ldg: 64 points, 3 regions 17.8 us a call for 16.7, near the posterior
// (16384 points) 110.6 for 110.1; with __restrict__ nowhere: 32 models 498 for 494.
#pragma once
#include <cuda_runtime.h>
#include <utility>

namespace fg21 {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                             Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace fg21
