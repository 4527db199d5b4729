// Launches of a chain of kernels on one stream that overlap their starts: a kernel launched with chain_launch may begin
// once every block of its predecessor has begun, and calls chain_wait before it touches anything the predecessors
// write or read; every kernel of a chain calls chain_next first.  Hides most of the 2-3 us between dependent launches.
// Loads of what a predecessor wrote must be plain ones: the compiler moves __ldg and loads through const __restrict__
// pointers above the wait.
// (Kernels whose blocks wait for one another are launched cooperatively instead and start the ordinary way.)
#pragma once

#include <cuda_runtime.h>

namespace lot {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t chain_launch(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

} // namespace lot
