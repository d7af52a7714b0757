// sp2_launch.cuh -- launches that overlap with the end of the kernel before
// them in the stream (programmatic dependent launch).
//
// A call of this library is a short chain of kernels (copy, predict, pass,
// reduce) that each take a few microseconds at small sink counts, so the gaps
// between them count.  A kernel of the chain may be brought onto the SMs as soon
// as the CTAs of the one before it have left them, and starts with grid_wait():
// it waits until that kernel has completed and its writes are visible.  The
// launch latency thus runs beside the end of the kernel before; nothing is read
// or written before the wait, so the order of all memory accesses is that of
// plain stream order (a kernel waits for its predecessor's completion, which has
// itself waited for its own).  Letting the next kernel in any earlier
// (griddepcontrol.launch_dependents) was slower: waiting CTAs take registers
// from CTAs that have yet to start (1000 sinks on 100003 sources: 182 us a step
// with plain launches, 218 with the trigger, 172 without).  Others: one sink on
// 131072 sources 20.6 -> 17.7 us, 61 sinks 45 -> 37 us, a block run of 4096
// particles (three kernels a block) 2.77 -> 1.94 ms.
#pragma once

#include <cuda_runtime.h>

namespace sp2 {

__device__ __forceinline__ void grid_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... Params, class... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), unsigned grid, unsigned threads, size_t smem,
                                     cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // reported here, and not once more by the next launch of some other context
    return e;
}

}  // namespace sp2
