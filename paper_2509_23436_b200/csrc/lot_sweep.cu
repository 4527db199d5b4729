// Sweep path of the LOT attention (Eq. (1)-(2), scaling form): any supported shape, float32 or bf16 tensors, token
// weights, key lengths, starting potentials.
//
// A problem (one side of one slice) is shared by a group of C thread blocks.  lot_build.cu has left the stabilised Gibbs
// kernel K_it = 2^(L_it + Gref_t - ref_i) in global memory in float32; each block keeps the first `srows` rows of its
// share in shared memory and the next ones in tensor memory (TENSOR; the rest stays in L2) and runs the iterations on them:
//   s_i = sum_t K_it w_t,   c_t = sum_i m_i K_it / s_i,   w_t <- target_t / c_t        (G_t = Gref_t + log2 w_t)
// two multiply-adds per entry and pass, no exponential and no logarithm.  Column sums are added lane -> warp -> block ->
// cluster -> group in a fixed order (group_columns).  When a weight leaves its range (lot_sweep.h) the kernel is rebuilt around
// the current potentials; when a column sum itself leaves float32's range that iteration is redone in the log domain
// (column maxima first), so any spread of the potentials is exact.
// What bounds a pass: the latency of rows in flight (16 warps an SM: 18 entries a clock and SM from shared memory, 26 with tensor
// memory) and, for C > 1, the exchange.  64 problems of 16384 rows at RP = 256, 20 iterations: this kernel 3410 us with rows in shared
// memory and L2, 49 blocks a problem and words exchanged through L2; 1883 with six problems at once, 24 blocks each in clusters of two.
// The call with that split, the one chosen, 3305 us; with 18 blocks a problem 3618, 28 3584, 32 3571 (clusters of four 3553, of eight
// 4097), 24 in clusters of four 3807.
#include "lot_chain.cuh"
#include "lot_sweep_core.cuh"

#include <mutex>

namespace lot {
namespace sweep {

// Closing update and results of problem p.  Out of line, and everything worked out again: nothing of the problem is live
// across recover() and this call, which would cost the iteration loop its registers (spills in it: a fifth slower).
template <typename T, int RP, int CPL, int THREADS, bool TENSOR>
__device__ __noinline__ void finish(const SweepArgs *ap, int p, int c)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const SweepArgs &a = *ap;
    const Shared S = carve<T, RP, THREADS>(smem, a.srows);
    Share R;
    const Problem P = locate<RP, CPL, THREADS>(a, p, c, R);
    const int tid = threadIdx.x;
    if (P.nv > 0) {
        const Lane<RP, CPL> L = make_lane<RP, CPL, THREADS>(S, a.tcols);
        u64 w[CPL / 2], acc[CPL / 2];
        load_weights<RP, CPL>(L, w);
        pass<RP, CPL, THREADS, TENSOR, true>(L, R, w, acc, a.inv[P.side] + (size_t)P.slice * P.n + P.row0);
    }
    if (c == 0 && tid < RP) {
        const double gl = S.gref[tid];
        const float wl = tid < a.r ? S.w[tid] : 0.f;
        a.w[P.side][(size_t)P.slice * RP + tid] = wl;
        a.gref[P.side][(size_t)P.slice * RP + tid] = gl;
        if (tid < a.r && a.g_out[P.side] != nullptr)
            a.g_out[P.side][(size_t)P.slice * a.r + tid] = (float)((gl + log2((double)wl)) * a.eps_ln2);
    }
}

// KEEP: the weights of every iteration go to a.hist (backward).
template <typename T, int RP, int CPL, int THREADS, bool GROUP, bool TENSOR, bool KEEP>
__global__ void __launch_bounds__(THREADS, max_blocks(CPL, THREADS))
sweep_kernel(const __grid_constant__ SweepArgs a)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, group = GROUP ? blockIdx.x / a.C : blockIdx.x, c = GROUP ? blockIdx.x % a.C : 0;
    const int NP = 2 * a.B * a.H, r = a.r;
    unsigned seq = a.seq0;
    const Shared S = carve<T, RP, THREADS>(smem, a.srows);
    if (tid == 0) { S.flag[0] = 0; S.flag[1] = 0; }
    if (GROUP) open_exchange<RP>(a, S);
    if (TENSOR) open_tensor(S, a.tcols);
    chain_wait();

    for (int p = group; p < NP; p += a.groups) {
        Share R;
        const Problem P = locate<RP, CPL, THREADS>(a, p, c, R);
        __syncthreads();                                     // the previous problem is done with shared memory
        if (tid < RP) {
            double g0 = -(double)kStartLog2;
            if (tid < r && a.g_in[P.side] != nullptr) g0 += (double)__ldg(a.g_in[P.side] + (size_t)P.slice * r + tid) * a.scale;
            S.gref[tid] = g0;
            S.w[tid] = tid < r ? kStart : 0.f;
            S.tgt[tid] = tid < r ? __ldg(a.beta + P.h * r + tid) * (R.mass ? 1.f : (float)P.nv) : 0.f;
        }
        load_rows<RP, CPL, THREADS>(S, R);
        if constexpr (TENSOR) load_tensor_rows<RP, CPL, THREADS>(S, R, a.tcols);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (P.nv <= 0 && tid == 0 && c == 0) atomicOr(a.status, 2 /* LOT_DEV_EMPTY */);
        __syncthreads();
        float wold = 0.f, wnew = S.w[tid < RP ? tid : 0];
        bool bad = false;
        int it = 0;
        if (P.nv > 0) {
            const Lane<RP, CPL> L = make_lane<RP, CPL, THREADS>(S, a.tcols);
            const float tgt = S.tgt[tid < RP ? tid : 0];
            u64 w[CPL / 2];
            load_weights<RP, CPL>(L, w);
            float *hp = KEEP && c == 0 && tid < RP ? a.hist + (size_t)p * RP + tid : nullptr;      // thread t's column
            if (KEEP && hp != nullptr) *hp = S.w[tid];
            for (; it < a.iters; ++it) {
                bad = iterate<RP, CPL, THREADS, GROUP, TENSOR>(a, S, R, L, w, tgt, group, c, seq, wold, wnew);
                if (bad) break;
                if (KEEP && hp != nullptr) {
                    hp += (size_t)NP * RP;
                    *hp = tid < r ? wnew : 0.f;
                }
            }
            if (KEEP && !bad && c == 0 && tid == 0) a.wide[p] = 0;
        }
        if (bad) seq = recover<T, RP, CPL, THREADS, GROUP, TENSOR>(&a, p, group, c, it, seq, wold, wnew);
        if (p + a.groups >= NP) chain_next();
        finish<T, RP, CPL, THREADS, TENSOR>(&a, p, c);
    }
    if (TENSOR) close_tensor(S, a.tcols);
    if (GROUP) close_exchange(a);
}

template <typename T, int RP, int CPL, int THREADS, bool GROUP, bool TENSOR, bool KEEP>
static cudaError_t launch_g(const SweepPlan &P, const SweepArgs &a, cudaStream_t st)
{
    auto kern = sweep_kernel<T, RP, CPL, THREADS, GROUP, TENSOR, KEEP>;
    if (P.tcols != 0 && P.smem < kAloneSmem) return cudaErrorInvalidConfiguration;
    static std::mutex mu;
    static bool attr_set[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!attr_set[dev]) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerBlock);
            if (e != cudaSuccess) return e;
            attr_set[dev] = true;
        }
    }
    const dim3 grid((unsigned)(P.groups * P.C));
    if (P.chained) return chain_launch(kern, grid, THREADS, P.smem, P.K, st, a);
    if (P.C == P.K) return cluster_launch(kern, grid, THREADS, P.smem, P.K, st, a);
    return group_launch(kern, grid, THREADS, P.smem, P.K, st, a);
}

template <typename T, int RP, bool KEEP>
static cudaError_t launch_k(const SweepPlan &P, const SweepArgs &a, cudaStream_t st)
{
    if constexpr (RP <= 32 && !KEEP) {
        if (P.threads == 32) return launch_g<T, RP, wide_cols(RP), 32, false, false, false>(P, a, st);
    }
    if (P.threads == kTensorThreads)
        return P.C > 1 ? launch_g<T, RP, kTensorLane, kTensorThreads, true, true, KEEP>(P, a, st)
                       : launch_g<T, RP, kTensorLane, kTensorThreads, false, true, KEEP>(P, a, st);
    return P.C > 1 ? launch_g<T, RP, wide_cols(RP), 256, true, false, KEEP>(P, a, st) : launch_g<T, RP, wide_cols(RP), 256, false, false, KEEP>(P, a, st);
}

template <typename T, bool KEEP>
static cudaError_t launch_rp(const SweepPlan &P, const SweepArgs &a, cudaStream_t st)
{
    switch (P.RP) {
    case 16: return launch_k<T, 16, KEEP>(P, a, st);
    case 32: return launch_k<T, 32, KEEP>(P, a, st);
    case 64: return launch_k<T, 64, KEEP>(P, a, st);
    case 128: return launch_k<T, 128, KEEP>(P, a, st);
    default: return launch_k<T, 256, KEEP>(P, a, st);
    }
}

#ifndef LOT_SWEEP_PART                                       // this file by itself: float32 tensors; the others are compiled side by side
cudaError_t launch_f32(const SweepPlan &P, const SweepArgs &a, cudaStream_t st) { return launch_rp<float, false>(P, a, st); }

int cluster_count(int K, size_t smem)
{
    auto kern = sweep_kernel<float, 16, wide_cols(16), 256, true, false, false>;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = K;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)K);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerBlock) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}
#endif

} // namespace sweep
} // namespace lot
