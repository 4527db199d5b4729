// The stabilised Gibbs kernel from bf16 tokens, more than 32 pivots, up to 128 channels: tcgen05 products with accumulators in
// tensor memory.  What it computes: lot_build.cu.
//
// A block belongs to a head: it stages the head's pivots once, as three (two) bf16 terms whose sum is exact, and goes through
// 128-token tiles of all batch rows and both sides.  While the products of one tile run (terms x d / 16 instructions of 128 x RP x 16, small
// terms first, one thread issues them) all warps turn the accumulators of the tile before into kernel rows, and the next tile's
// tokens are on their way into registers: two threads share a row (four measured no faster).
// Bound by the write of the kernel (4 bytes an entry).  With warp-level products every warp read all pivots' terms from shared
// memory for 16 tokens (75% of its bandwidth, tensor cores at 39%): B = 4, H = 8, n = 16384, d = 128, r = 256, 1.07 GB of kernel,
// 985 us, now 388; 16 x 17 tiles of d = 128, r = 256 36 us, now 24; n = 4096, H = 16, d = 64, r = 64 24 us, now 20.  The potentials' error
// against float64 is half of what it was (rms in units of eps at d = 128, r = 256: 8e-7, before 2e-6).
// Taken however few the tiles are: at r <= 64, d <= 64 and fewer than 400 tiles a call is up to 2 us slower than with warp-level products
// (16 slices of 120 tokens 24.8 us, 22.9; 64 of 384 43.3, 41.3; faster from 512 tiles on, and nearly everywhere at d = 128 or r > 64), but its
// potentials have two thirds of the error there too (16 slices of 64 tokens at r = 64 9.7e-7 and 1.5e-6 of eps).
#include "lot_chain.cuh"
#include "lot_internal.h"
#include "lot_logits.cuh"
#include "lot_sm100.cuh"
#include "lot_sweep.h"

#include <mutex>

namespace lot {
namespace build_tc {

using namespace sm100;
constexpr int kThreads = 256, kTile = 128;

struct Layout {
    int kb;                  // blocks of 64 channels
    int offX, offG, offMax, offBar, total;
};
__host__ __device__ inline Layout layout(int RP, int d, int terms)
{
    Layout L;
    L.kb = (d + 63) / 64;
    L.offX = terms * L.kb * RP * 128;
    L.offG = L.offX + L.kb * kTile * 128;
    L.offMax = L.offG + RP * 4;
    L.offBar = L.offMax + kThreads * 4;
    L.total = L.offBar + 32;
    return L;
}

// Behind it the 32 columns just requested may be used.
__device__ __forceinline__ void settle(float (&v)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]), "+f"(v[8]), "+f"(v[9]), "+f"(v[10]),
                   "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]), "+f"(v[15])::"memory");
    asm volatile("" : "+f"(v[16]), "+f"(v[17]), "+f"(v[18]), "+f"(v[19]), "+f"(v[20]), "+f"(v[21]), "+f"(v[22]), "+f"(v[23]), "+f"(v[24]), "+f"(v[25]),
                   "+f"(v[26]), "+f"(v[27]), "+f"(v[28]), "+f"(v[29]), "+f"(v[30]), "+f"(v[31])::"memory");
}

// A whole 32-byte sector by one thread: its row's neighbours belong to other lines.
__device__ __forceinline__ void store8(float *p, const float *v)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]),
                 "f"(v[6]), "f"(v[7]) : "memory");
}

struct Tile {
    int slice, side, row0, rows;
};

template <int RP>
__global__ void __launch_bounds__(kThreads, RP == 256 ? 1 : 2)
build_tc_kernel(const __grid_constant__ SweepArgs a, int tiles_q, int tiles_k, int per_head)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int PARTS = kThreads / kTile, COLS = RP / PARTS, NX = 2 * 8 * kTile / kThreads;        // threads a row, their columns, 16-byte chunks a thread fetches
    const Layout L = layout(RP, a.d, a.terms);
    const uint32_t sbase = smem_u32(smem), bar = sbase + L.offBar;
    float *sG = reinterpret_cast<float *>(smem + L.offG), *sMax = reinterpret_cast<float *>(smem + L.offMax);
    volatile int *sAbort = reinterpret_cast<volatile int *>(smem + L.offBar + 8);
    uint32_t *sTmem = reinterpret_cast<uint32_t *>(smem + L.offBar + 16);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, r = a.r, d = a.d;
    const int h = blockIdx.x / per_head, first = blockIdx.x % per_head, both = tiles_q + tiles_k;
    if ((sbase & 1023u) != 0) { if (tid == 0) atomicOr(a.status, 4); return; }
    // what the later kernels of the call count and flag in starts at zero
    for (size_t i = (size_t)blockIdx.x * kThreads + tid; i < a.head_words; i += (size_t)gridDim.x * kThreads) a.head[i] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        mbar_init(bar, 1);
        *sAbort = 0;
        fence_barrier_init();
    }
    if (warp == 0) { tmem_alloc(smem_u32(sTmem), 2 * RP); tmem_relinquish(); }
    // pivots: rows of 128 bytes, 16-byte chunks permuted by the row (128-byte swizzle), planes [term][64 channels][RP rows]
    const float *z = a.z + (size_t)h * r * d;
    for (int idx = tid; idx < RP * L.kb * 8; idx += kThreads) {
        const int t = idx % RP, ck = idx / RP, c = ck * 8;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = 0.f;
        if (t < r && c < d) {
            const float4 x = __ldg(reinterpret_cast<const float4 *>(z + (size_t)t * d + c)), y = __ldg(reinterpret_cast<const float4 *>(z + (size_t)t * d + c + 4));
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
        }
        uint32_t o[4][3];
#pragma unroll
        for (int e = 0; e < 4; ++e) logits::split<3>(v[2 * e], v[2 * e + 1], o[e]);
#pragma unroll
        for (int term = 0; term < 3; ++term)
            if (term < a.terms)
                *reinterpret_cast<uint4 *>(smem + (size_t)((term * L.kb + ck / 8) * RP + t) * 128 + (((ck & 7) ^ (t & 7)) << 4)) =
                    make_uint4(o[0][term], o[1][term], o[2][term], o[3][term]);
    }
    for (int t = tid; t < RP; t += kThreads) sG[t] = t < r ? 0.f : neg_inf();

    auto tile = [&](int w) {
        Tile T;
        const int b = w / both, rest = w % both;
        T.side = rest < tiles_k ? 1 : 0;
        T.slice = b * a.H + h;
        T.row0 = (T.side ? rest : rest - tiles_k) * kTile + a.skip;
        int nv = a.n[T.side];
        if (T.side == 1 && a.key_len != nullptr) nv = min(max(__ldg(a.key_len + b), 0), nv);
        T.rows = min(nv - T.row0, kTile);                    // rows without mass are never read
        return T;
    };
    auto find = [&](int w) {                                 // the first place of the head's list from w on whose tile has rows, or -1
        for (; w < a.B * both; w += per_head)
            if (tile(w).rows > 0) return w;
        return -1;
    };
    uint4 x[NX];                                             // chunk u of the tile: row idx % 128, chunk idx / 128
    auto fetch = [&](const Tile &T) {
        const __nv_bfloat16 *p = static_cast<const __nv_bfloat16 *>(a.x[T.side]) + ((size_t)T.slice * a.n[T.side] + T.row0) * d;
#pragma unroll
        for (int u = 0; u < NX; ++u) {
            if (u * kThreads >= 8 * L.kb * kTile) break;
            const int idx = tid + u * kThreads, chunk = idx % (8 * L.kb), row = idx / (8 * L.kb);
            x[u] = row < T.rows && chunk * 8 < d ? __ldg(reinterpret_cast<const uint4 *>(p + (size_t)row * d + chunk * 8)) : make_uint4(0, 0, 0, 0);
        }
    };
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *sTmem;
    constexpr uint32_t idesc = make_idesc_bf16(128, RP, 0, 0);
    const uint64_t desc = make_smem_desc(sbase, 16, 1024);
    const uint32_t d_hi = (uint32_t)(desc >> 32), d_lo = (uint32_t)desc;

    int at = find(first);
    if (at >= 0) fetch(tile(at));
    int before = -1;
    for (int i = 0; at >= 0 || before >= 0; ++i) {
        if (i > 0) mbar_wait(bar, (i - 1) & 1, sAbort, a.status);                 // the products of the tile before
        const int now = at;
        if (now >= 0) {
#pragma unroll
            for (int u = 0; u < NX; ++u) {
                if (u * kThreads >= 8 * L.kb * kTile) break;
                const int idx = tid + u * kThreads, chunk = idx % (8 * L.kb), row = idx / (8 * L.kb);
                *reinterpret_cast<uint4 *>(smem + L.offX + (size_t)((chunk >> 3) * kTile + row) * 128 + (((chunk & 7) ^ (row & 7)) << 4)) = x[u];
            }
            fence_proxy_async_smem();
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            if (warp == 0 && elect_one()) {
                const uint32_t acc = tmem + (i & 1) * RP;
                bool more = false;
                for (int term = a.terms - 1; term >= 0; --term)
                    for (int ks = 0; ks * 16 < d; ++ks) {
                        const uint32_t xa = d_lo + ((L.offX + (ks >> 2) * kTile * 128) >> 4) + (ks & 3) * 2;
                        const uint32_t za = d_lo + (((term * L.kb + (ks >> 2)) * RP * 128) >> 4) + (ks & 3) * 2;
                        umma_bf16(acc, ((uint64_t)d_hi << 32) | xa, ((uint64_t)d_hi << 32) | za, idesc, more ? 1u : 0u);
                        more = true;
                    }
                umma_commit(bar);
            }
            __syncwarp();
            at = find(at + per_head);
            if (at >= 0) fetch(tile(at));
        }
        if (before >= 0) {
            if (now < 0) {
                chain_next();
                __syncthreads();                             // else the barrier above: the exchange below has been read
            }
            const Tile T = tile(before);
            if (a.g_in[0] != nullptr || a.g_in[1] != nullptr) {
                const float *g = a.g_in[T.side];
                for (int t = tid; t < r; t += kThreads) sG[t] = g ? (float)((double)__ldg(g + (size_t)T.slice * r + t) * a.scale) : 0.f;
                __syncthreads();
            }
            tc_fence_after();
            const int row = (warp & 3) * 32 + lane, part = warp >> 2;
            const uint32_t acc = tmem + ((uint32_t)((warp & 3) * 32) << 16) + ((i - 1) & 1) * RP + part * COLS;
            const float scale = (float)a.scale;
            const float4 *G = reinterpret_cast<const float4 *>(sG + part * COLS);
            float m = neg_inf();
#pragma unroll
            for (int c = 0; c < COLS; c += 32) {
                float v[32];
                tmem_ld32(acc + c, v);
                settle(v);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float4 gg = G[c / 4 + e];
                    m = fmaxf(m, fmaxf(fmaxf(fmaf(v[4 * e], scale, gg.x), fmaf(v[4 * e + 1], scale, gg.y)), fmaxf(fmaf(v[4 * e + 2], scale, gg.z), fmaf(v[4 * e + 3], scale, gg.w))));
                }
            }
            sMax[part * kTile + row] = m;
            __syncthreads();
#pragma unroll
            for (int o = 0; o < PARTS; ++o) m = fmaxf(m, sMax[o * kTile + row]);
            m -= kKernelTop;
            float *o = a.kt[T.side] + ((size_t)T.slice * a.n[T.side] + T.row0 + row) * RP + part * COLS;
#pragma unroll
            for (int c = 0; c < COLS; c += 32) {
                float v[32];
                tmem_ld32(acc + c, v);
                settle(v);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float4 gg = G[c / 4 + e];
                    v[4 * e] = ex2(fmaf(v[4 * e], scale, gg.x) - m);
                    v[4 * e + 1] = ex2(fmaf(v[4 * e + 1], scale, gg.y) - m);
                    v[4 * e + 2] = ex2(fmaf(v[4 * e + 2], scale, gg.z) - m);
                    v[4 * e + 3] = ex2(fmaf(v[4 * e + 3], scale, gg.w) - m);
                }
                if (row < T.rows) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) store8(o + c + 8 * e, v + 8 * e);
                }
            }
        }
        before = now;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, 2 * RP);
}

template <int RP>
static cudaError_t launch_t(const SweepArgs &a, cudaStream_t st)
{
    auto kern = build_tc_kernel<RP>;
    const Layout L = layout(RP, a.d, a.terms);
    static std::mutex mu;
    static bool attr_set[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!attr_set[dev]) {
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, layout(RP, 128, 3).total);
            if (e != cudaSuccess) return e;
            attr_set[dev] = true;
        }
    }
    // blocks an SM holds (registers, accumulators, shared memory), shared evenly by the heads
    const int fit = RP < 256 && 2 * (L.total + 1024) <= 228 * 1024 ? 2 : 1, slots = fit * device_sm_count();
    const int tq = (a.n[0] - a.skip + kTile - 1) / kTile, tk = (a.n[1] - a.skip + kTile - 1) / kTile;
    const int tiles = a.B * (tq + tk), share = slots / a.H < 1 ? 1 : slots / a.H;
    const int per_head = tiles < share ? (tiles < 1 ? 1 : tiles) : share;
    kern<<<(unsigned)(per_head * a.H), kThreads, L.total, st>>>(a, tq, tk, per_head);
    return cudaGetLastError();
}

} // namespace build_tc

bool build_tc_supported(int RP, int d) { return RP >= 64 && d <= 128; }

cudaError_t launch_build_tc(int RP, const SweepArgs &a, cudaStream_t st)
{
    using namespace build_tc;
    return RP == 64 ? launch_t<64>(a, st) : RP == 128 ? launch_t<128>(a, st) : launch_t<256>(a, st);
}

} // namespace lot
