// The stabilised Gibbs kernel of the sweep path (lot_sweep.cu) from tokens and pivots: logits, row maxima, exponentials in
// one kernel; every warp holds whole rows of logits in its accumulators.  bf16 tokens with more than 32 pivots and up to 128
// channels: lot_build_tc.cu.
#include "lot_chain.cuh"
#include "lot_internal.h"
#include "lot_logits.cuh"
#include "lot_sweep.h"

#include <mutex>

namespace lot {
namespace build {

constexpr int kThreads = 256, kWarps = 8;

template <typename T, int RP> struct Shape {
    static constexpr int ROWS = sizeof(T) == 4 && RP == 256 ? 8 : 16;                    // per warp
    static constexpr int ACC = (RP / 8) * (ROWS / 8) * 2 * (sizeof(T) == 4 ? 2 : 1);     // accumulator registers
    static constexpr int MINB = ACC <= 32 ? 3 : ACC <= 64 ? 2 : 1;
};

template <typename T, int RP, int TERMS>
__global__ void __launch_bounds__(kThreads, Shape<T, RP>::MINB)
build_kernel(const __grid_constant__ SweepArgs a, int tiles_q, int tiles_k)
{
    extern __shared__ __align__(128) uint8_t stage[];
    typedef Shape<T, RP> Sh;
    typedef logits::Logits<T, RP, Sh::ROWS, kThreads, TERMS> Lg;
    typedef typename Lg::LT LT;
    __shared__ LT sG[RP];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3, r = a.r;
    const int both = tiles_q + tiles_k, slice = blockIdx.x / both, rest = blockIdx.x % both;
    const int side = rest < tiles_k ? 1 : 0, tile = side ? rest : rest - tiles_k;
    const int b = slice / a.H, h = slice % a.H, n = a.n[side];
    int nv = n;
    if (side == 1 && a.key_len != nullptr) nv = min(max(__ldg(a.key_len + b), 0), n);
    // what the later kernels of the call count and flag in starts at zero
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < a.head_words; i += (size_t)gridDim.x * kThreads) a.head[i] = make_uint4(0, 0, 0, 0);
    const int row0 = tile * (kWarps * Sh::ROWS) + a.skip;
    if (row0 >= nv) return;                                        // rows without mass are never read
    if (threadIdx.x < RP) {
        LT g0 = (LT)0;
        if ((int)threadIdx.x < r && a.g_in[side] != nullptr) g0 = (LT)((double)__ldg(a.g_in[side] + (size_t)slice * r + threadIdx.x) * a.scale);
        sG[threadIdx.x] = g0;
    }
    const int w0 = row0 + warp * Sh::ROWS, wrows = min(max(nv - w0, 0), Sh::ROWS);
    Lg lg;
    lg.run(static_cast<const T *>(a.x[side]) + ((size_t)slice * n + w0) * a.d, wrows, a.d, a.z + (size_t)h * r * a.d, r, stage, lane);
    chain_next();
    float *kt = a.kt[side] + ((size_t)slice * n + w0) * RP;
#pragma unroll
    for (int hh = 0; hh < Sh::ROWS / 8; ++hh) {
        LT m = (LT)neg_inf();
#pragma unroll
        for (int j = 0; j < RP / 8; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int t = 8 * j + 2 * q + e;
                const LT l = t < r ? fma(lg.at(j, hh, e), (LT)a.scale, sG[t]) : (LT)neg_inf();
                lg.at(j, hh, e) = l;
                m = fmax(m, l);
            }
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, 2));
        m -= (LT)kKernelTop;
        const int i = g + 8 * hh;
        if (i < wrows) {
#pragma unroll
            for (int j = 0; j < RP / 8; ++j) {
                const float2 v = make_float2(ex2((float)(lg.at(j, hh, 0) - m)), ex2((float)(lg.at(j, hh, 1) - m)));
                *reinterpret_cast<float2 *>(kt + (size_t)i * RP + 8 * j + 2 * q) = v;
            }
        }
    }
}

template <typename T, int RP, int TERMS = 3>
static cudaError_t launch_t(const SweepArgs &a, cudaStream_t st)
{
    typedef Shape<T, RP> Sh;
    auto kern = build_kernel<T, RP, TERMS>;
    constexpr size_t smem = logits::stage_bytes<T>(RP);
    if (smem > 48 * 1024) {
        static std::mutex mu;
        static bool attr_set[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(mu);
        if (!attr_set[dev]) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            attr_set[dev] = true;
        }
    }
    constexpr int rows = kWarps * Sh::ROWS;
    const int tq = (a.n[0] + rows - 1) / rows, tk = (a.n[1] + rows - 1) / rows;
    kern<<<(unsigned)((tq + tk) * a.B * a.H), kThreads, smem, st>>>(a, tq, tk);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_rp(int RP, const SweepArgs &a, cudaStream_t st)
{
    switch (RP) {
    case 16: return launch_t<T, 16>(a, st);
    case 32: return launch_t<T, 32>(a, st);
    case 64: return launch_t<T, 64>(a, st);
    case 128: return launch_t<T, 128>(a, st);
    default: return launch_t<T, 256>(a, st);
    }
}

} // namespace build

cudaError_t launch_build(int RP, const SweepArgs &a, int dtype, cudaStream_t st)
{
    if (dtype == 1 && build_tc_supported(RP, a.d)) return launch_build_tc(RP, a, st);       // whatever the number of tiles: lot_build_tc.cu
    if (dtype == 1 && a.terms == 2) {
        if (RP == 16) return build::launch_t<__nv_bfloat16, 16, 2>(a, st);
        if (RP == 32) return build::launch_t<__nv_bfloat16, 32, 2>(a, st);
    }
    return dtype == 0 ? build::launch_rp<float>(RP, a, st) : build::launch_rp<__nv_bfloat16>(RP, a, st);
}

} // namespace lot
