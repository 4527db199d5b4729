// Launches of a chain of kernels on one stream that overlap their starts: a kernel launched with chain_launch may begin
// once every block of its predecessor has called chain_next or ended, and calls chain_wait before it touches anything
// the predecessors write or read.  Every path through such a kernel passes chain_wait, also of one that touches nothing of
// theirs (it waits last): the end of the last kernel is taken for the end of the chain.  chain_next stands where a block's main work is done: called first thing, the waiting
// blocks of the next kernel took a fifth of the sweep kernel's speed.  Hides most of the 2-3 us between dependent launches.
// Loads of what a predecessor wrote must be plain ones: the compiler moves __ldg and loads through const __restrict__
// pointers above the wait.
// (Kernels whose blocks wait for blocks of other clusters are launched cooperatively instead and start the ordinary way.)
#pragma once

#include <cuda_runtime.h>

namespace lot {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Loads that stay below the wait (and coherent ones: the read-only path may hold lines from before it).
__device__ __forceinline__ float4 chain_ld4(const float *p)
{
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 chain_ld2(const float *p)
{
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float chain_ld(const float *p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// A launch in clusters of K blocks with one more attribute, or none (attr.id == cudaLaunchAttributeIgnore).
template <typename... P, typename... A>
inline cudaError_t launch_with(cudaLaunchAttribute attr, void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, int K, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2] = {attr, {}};
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)K;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = K > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

template <typename... P, typename... A>
inline cudaError_t chain_launch(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, int K, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    return launch_with(at, kern, grid, threads, smem, K, st, args...);
}
template <typename... P, typename... A>
inline cudaError_t chain_launch(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A... args)
{
    return chain_launch(kern, grid, threads, smem, 1, st, args...);
}

// The ordinary start, in clusters of K.
template <typename... P, typename... A>
inline cudaError_t cluster_launch(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, int K, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeIgnore;
    return launch_with(at, kern, grid, threads, smem, K, st, args...);
}

// A kernel whose blocks wait for one another across clusters: all of them run at once.  Blocks that wait only within their cluster do not need
// it, the hardware starts a cluster whole; a cooperative launch starts the ordinary way, and ncu gives no time for one in clusters.
template <typename... P, typename... A>
inline cudaError_t group_launch(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, int K, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    return launch_with(at, kern, grid, threads, smem, K, st, args...);
}

} // namespace lot
