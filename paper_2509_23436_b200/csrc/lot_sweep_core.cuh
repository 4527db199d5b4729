// Device code shared by the sweep kernels (lot_sweep.cu: forward, lot_sweep_bwd.cu: reverse): how a problem lies over blocks,
// lanes and shared memory, passes over the stored Gibbs kernel, column reductions, the exchange between the blocks of
// a group, and the kernel's rebuilding.
#pragma once

#include "lot_common.cuh"
#include "lot_internal.h"
#include "lot_logits.cuh"
#include "lot_sm100.cuh"
#include "lot_sweep.h"

#include <math.h>
#include <string.h>

namespace lot {
namespace sweep {

typedef unsigned long long u64;
using sm100::global_timer_ns;

__host__ __device__ constexpr int kTileRows(int threads) { return threads / 2; }   // 16 rows per warp
constexpr float kLostLo = 1e-30f, kLostHi = 1e38f;
constexpr float kFarLo = 7.7037198e-34f, kFarHi = 1.1258999e15f;   // 2^-110, 2^50
constexpr float kStart = 8.8817842e-16f;                            // 2^kStartLog2
constexpr float kHistLo = 2.4074124e-35f, kHistHi = 4.1538374e34f;   // 2^-115, 2^115: kept weights a reverse pass can use
constexpr int kPeers = 8, kWords = 16;                               // blocks of a cluster (the portable limit); words a thread waits for at once
constexpr int kSmPerBlockReserve = 1024, kSmemPerSM = 228 * 1024, kSmemPerBlock = 227 * 1024;
constexpr unsigned long long kWaitNs = 1000000000ull;

// floats <-> packed pairs for fma.rn.f32x2
__device__ __forceinline__ u64 pack_f2(float lo, float hi)
{
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack_f2(u64 v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ u64 fma_f2(u64 a, u64 b, u64 c)
{
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void lds2(u64 &a, u64 &b, uint32_t addr)
{
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}
__device__ __forceinline__ float lds(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }

// A row of RP columns lies over LPR = RP / CPL adjacent lanes, CPL columns (CPL / 4 chunks of 16 bytes) per lane: chunk v of
// lane cl is v * LPR + cl.  In shared memory the chunks of a row are permuted so that the eight lanes of a 128-byte phase, which
// cover 8 / LPR rows, fall on different banks; a row starts at a multiple of its length there (the area is aligned to 1024 bytes).
template <int RP, int CPL> struct Lay {
    static constexpr int LPR = RP / CPL, RPW = 32 / LPR, CH = RP / 4, NV = CPL / 4;
    static constexpr int RPL = RP >= 32 ? 1 : 32 / RP, SG = LPR >= 8 ? 1 : (8 / LPR / RPL < 1 ? 1 : 8 / LPR / RPL);
    static __device__ __forceinline__ int swz(int row, int chunk) { return chunk ^ (((row / RPL) & (SG - 1)) * LPR); }
};

// columns per lane where a pass is bound by issue and shared-memory reads, not by latency
__host__ __device__ constexpr int wide_cols(int RP) { return RP <= 32 ? 8 : 16; }

// blocks per SM that the registers allow (80 a thread, 128 with sixteen columns per lane)
__host__ __device__ constexpr int max_blocks(int cpl, int threads) { return (cpl == 16 ? 512 : 768) / threads; }

// Blocks that keep rows in tensor memory too: twice the threads, sixteen columns a lane whatever RP is, all of the SM's columns.  Two of
// them on one SM would wait for each other, one in tcgen05.alloc, which no limit ends, the other for its column sums.  So such a
// block takes more than half of the SM's shared memory, whatever it needs (plans and launches hold to it).  Registers would not do: 512
// threads have all of them only as long as the compiler uses more than 64 a thread.
constexpr int kTensorThreads = 512, kTensorCols = 512, kTensorLane = 16;
constexpr size_t kAloneSmem = kSmemPerSM / 2;
static_assert(2 * (kAloneSmem + kSmPerBlockReserve) > (size_t)kSmemPerSM && kAloneSmem <= (size_t)kSmemPerBlock, "one such block an SM");
__host__ __device__ constexpr int lane_sharers(int threads) { return threads < 128 ? 1 : threads / 128; }       // warps that share a quarter of the lanes

// shared memory: [kernel rows | gref | work area (staged pivots, or the column reduction) | refs | weights, targets | flags,
// barriers | columns from the blocks of the cluster]
__host__ __device__ constexpr int rebuild_cols(int RP) { return RP < 32 ? RP : 32; }      // columns per step of a rebuild
template <typename T> __host__ __device__ constexpr size_t work_bytes(int RP, int threads)
{
    const size_t red = (size_t)(threads / 32) * RP * 4, st = logits::stage_bytes<T>(rebuild_cols(RP));
    return red > st ? red : st;
}
__host__ __device__ constexpr size_t ref_bytes(int RP, int threads)
{
    const size_t refs = (size_t)kTileRows(threads) * (RP / rebuild_cols(RP)) * 4, cols = (size_t)threads * 4;
    return refs > cols ? refs : cols;
}
template <typename T> __host__ __device__ constexpr size_t fixed_bytes(int RP, int threads)
{
    return work_bytes<T>(RP, threads) + ref_bytes(RP, threads) + (size_t)RP * (4 + 4 + 8) + 64;
}

struct Shared {
    float *K;                // kernel rows; up to a multiple of the block's rows per step, the last ones zero
    uint8_t *work;
    float *ref, *w, *tgt;
    double *gref;
    volatile int *flag;      // [0] a wait gave up, [1] a weight left its range
    uint32_t bars, peers;    // addresses of two barriers, and of what they count (group_columns)
    uint32_t tmem;           // address of the word that holds the tensor memory's address
};

// A block's share of one problem.
struct Share {
    float *g;                // its rows in global memory, [nrows][RP], or nullptr (all of them are in shared memory)
    const float *mass;       // its tokens' weights or nullptr
    int nrows, ns, steps;    // rows, of which the first ns are in shared memory too, in `steps` steps of the block
    int nt, tsteps;          // ... the next nt in tensor memory, in `tsteps` steps (an even number)
};

template <int RP, int CPL> __device__ __forceinline__ float4 *chunk_ptr(const Shared &S, const Share &R, int i, int chunk)
{
    return i < R.ns ? reinterpret_cast<float4 *>(S.K + (size_t)i * RP) + Lay<RP, CPL>::swz(i, chunk)
                    : reinterpret_cast<float4 *>(R.g + (size_t)i * RP) + chunk;
}

// The block's kernel rows again, around the reference potentials S.gref: exponents e_it = L_it + Gref_t - max_t(.) (EXPS),
// or the kernel.  Columns come in chunks of 32, which keeps the accumulators few beside the pass's registers: a chunk is
// stored relative to its own maximum first (the float32 rounding of an exponent must not depend on far-away columns)
// and the chunks of a row are combined in a second sweep.  Rare: see the exponent range in lot_sweep.h.
template <typename T, int RP, int CPL, int THREADS, bool EXPS>
__device__ __forceinline__ void build(const Shared &S, const Share &R, const T *x, const float *z, int d, int r, double scale)
{
    constexpr int CC = rebuild_cols(RP), NCH = RP / CC, ROWS = kTileRows(THREADS);
    typedef logits::Logits<T, CC, 16, THREADS> Lg;
    typedef typename Lg::LT LT;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
    for (int rt = 0; rt < R.nrows; rt += ROWS) {
        const int w0 = rt + warp * 16, wrows = min(max(R.nrows - w0, 0), 16);
#pragma unroll 1
        for (int ch = 0; ch < NCH; ++ch) {
            Lg lg;
            lg.run(x + (size_t)w0 * d, wrows, d, z + (size_t)ch * CC * d, min(max(r - ch * CC, 0), CC), S.work, lane);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                LT m = (LT)neg_inf();
#pragma unroll
                for (int j = 0; j < CC / 8; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int t = ch * CC + 8 * j + 2 * q + e;
                        const LT l = t < r ? fma(lg.at(j, h, e), (LT)scale, (LT)S.gref[t]) : (LT)neg_inf();
                        lg.at(j, h, e) = l;
                        m = fmax(m, l);
                    }
                m = fmax(m, __shfl_xor_sync(0xffffffffu, m, 1));
                m = fmax(m, __shfl_xor_sync(0xffffffffu, m, 2));
                const float mf = (float)m;
                const int i = w0 + g + 8 * h;
                if (NCH > 1 && q == 0) S.ref[(warp * 16 + g + 8 * h) * NCH + ch] = mf;
                if (i < R.nrows) {
#pragma unroll
                    for (int j = 0; j < CC / 8; ++j) {
                        float2 v;
                        v.x = mf == neg_inf() ? neg_inf() : (float)(lg.at(j, h, 0) - (LT)mf);
                        v.y = mf == neg_inf() ? neg_inf() : (float)(lg.at(j, h, 1) - (LT)mf);
                        if (NCH == 1 && !EXPS) { v.x = ex2(v.x + kKernelTop); v.y = ex2(v.y + kKernelTop); }
                        const int c0 = ch * CC + 8 * j + 2 * q;
                        float *p = reinterpret_cast<float *>(chunk_ptr<RP, CPL>(S, R, i, c0 >> 2)) + (c0 & 3);
                        *reinterpret_cast<float2 *>(p) = v;
                        if (NCH == 1 && !EXPS && R.g != nullptr && i < R.ns) *reinterpret_cast<float2 *>(R.g + (size_t)i * RP + c0) = v;
                    }
                }
            }
        }
        if (NCH > 1) {
            __syncwarp();
            for (int i = w0; i < w0 + wrows; ++i) {
                const float *rf = S.ref + (i - rt) * NCH;
                float M = rf[0];
#pragma unroll
                for (int c = 1; c < NCH; ++c) M = fmaxf(M, rf[c]);
                for (int ck = lane; ck < RP / 4; ck += 32) {
                    float4 *p = chunk_ptr<RP, CPL>(S, R, i, ck);
                    const float off = rf[ck / (CC / 4)] - M + (EXPS ? 0.f : kKernelTop);
                    float4 v = *p;
                    v.x += off; v.y += off; v.z += off; v.w += off;
                    if (!EXPS) { v.x = ex2(v.x); v.y = ex2(v.y); v.z = ex2(v.z); v.w = ex2(v.w); }
                    *p = v;
                    if (!EXPS && R.g != nullptr && i < R.ns) reinterpret_cast<float4 *>(R.g + (size_t)i * RP)[ck] = v;
                }
            }
        }
    }
    __syncthreads();
}

__device__ __forceinline__ float group_sum(float v, int lpr)
{
    for (int off = lpr / 2; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

__device__ __forceinline__ float rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int CPL> struct Row { u64 k[CPL / 2]; };       // a lane's columns of a row

// One row's step of a pass: row sum against the weights, its reciprocal (times the token's weight), column sums.  A row of
// zeros adds nothing.
template <int RP, int CPL, bool SUMS>
__device__ __forceinline__ float row_step(const Row<CPL> &k, const u64 (&w)[CPL / 2], u64 (&acc)[CPL / 2], float mass)
{
    u64 s0 = 0, s1 = 0;
#pragma unroll
    for (int j = 0; j < CPL / 2; j += 2) { s0 = fma_f2(k.k[j], w[j], s0); s1 = fma_f2(k.k[j + 1], w[j + 1], s1); }
    float a, b, c, e;
    unpack_f2(s0, a, b);
    unpack_f2(s1, c, e);
    float s = (a + b) + (c + e);
#pragma unroll
    for (int off = Lay<RP, CPL>::LPR / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    const float inv = rcp(fmaxf(s, 1e-37f)) * mass;
    if (SUMS) {
        const u64 ii = pack_f2(inv, inv);
#pragma unroll
        for (int j = 0; j < CPL / 2; ++j) acc[j] = fma_f2(k.k[j], ii, acc[j]);
    }
    return inv;
}

// What a thread needs in every iteration, worked out once per problem: shared-memory addresses of its columns of its
// first row, of its weights and of the column it owns.
template <int RP, int CPL> struct Lane {
    uint32_t k[CPL / 4], w, red, own, t;
    int i0, cl;
    // Chunk v of the row `row` bytes (whole steps) behind the first.  ONE: from the first chunk's address alone (the permutation is an
    // exclusive or within the row), an instruction more and three registers fewer: for the passes beside tensor memory, whose 128
    // registers do not hold everything, at r <= 32 (13376 x 7341 tokens, 12 slices, r = 32, T = 50: 254.3 us, 258.1 with four addresses).  At
    // r = 64 the instruction costs more than the reloads it saves (32 slices of 16384 tokens, T = 20: 975, 941).
    // Reloads of spilled registers a warp and pass, by local memory requests of 5 and 25 iterations: none at r <= 32, 3 to 9 of 260 to 400
    // instructions at r = 64, 1 at r = 256; the backward's forward 5 and its reverse steps 2, whatever the rows.
    template <bool ONE> __device__ __forceinline__ uint32_t chunk(uint32_t row, int v) const
    {
        return ONE ? (k[0] + row) ^ (v * (Lay<RP, CPL>::LPR * 16)) : k[v] + row;
    }
};

// The tensor memory as a second store of kernel rows: a lane's columns of a row are CPL neighbouring columns of its lane there, as
// it holds them in registers, so a warp only ever reads back what it has written itself (no operand layout, no bank
// conflicts).  The two warps that share a quarter of the lanes take half of the block's columns each.
template <int THREADS> __device__ __forceinline__ uint32_t tensor_rows(const Shared &S, int tcols)
{
    uint32_t base;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(base) : "r"(S.tmem) : "memory");
    const uint32_t warp = threadIdx.x >> 5;
    return base + ((warp & 3) << 21) + (warp >> 2) * (tcols / lane_sharers(THREADS));
}
// N = 16 or 32 columns of the lane as packed pairs; to be used behind settle().
template <int N> __device__ __forceinline__ void tensor_load(u64 (&v)[N / 2], uint32_t t)
{
    float f[N];
    sm100::tmem_ld<N>(t, f);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) v[i] = pack_f2(f[2 * i], f[2 * i + 1]);
}
template <int N> __device__ __forceinline__ void tensor_settle(u64 (&v)[N / 2])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+l"(v[0]), "+l"(v[1]), "+l"(v[2]), "+l"(v[3]), "+l"(v[4]), "+l"(v[5]), "+l"(v[6]), "+l"(v[7]) :: "memory");
    if constexpr (N == 32)                                   // the same wait stands for the other half
        asm volatile("" : "+l"(v[8]), "+l"(v[9]), "+l"(v[10]), "+l"(v[11]), "+l"(v[12]), "+l"(v[13]), "+l"(v[14]), "+l"(v[15]) :: "memory");
}
__device__ __forceinline__ void tensor_store16(uint32_t t, const float4 (&v)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(t), "f"(v[0].x), "f"(v[0].y), "f"(v[0].z), "f"(v[0].w), "f"(v[1].x), "f"(v[1].y), "f"(v[1].z), "f"(v[1].w), "f"(v[2].x),
                   "f"(v[2].y), "f"(v[2].z), "f"(v[2].w), "f"(v[3].x), "f"(v[3].y), "f"(v[3].z), "f"(v[3].w) : "memory");
}
// Rows ns .. ns + nt - 1 of the share from global into tensor memory, zeros up to the last step.
template <int RP, int CPL, int THREADS> __device__ __forceinline__ void load_tensor_rows(const Shared &S, const Share &R, int tcols)
{
    typedef Lay<RP, CPL> Y;
    static_assert(CPL == 16, "a row's part is sixteen columns");
    constexpr int STEP = (THREADS / 32) * Y::RPW;
    if (R.tsteps == 0) return;
    const int lane = threadIdx.x & 31, cl = lane % Y::LPR, i0 = (threadIdx.x >> 5) * Y::RPW + lane / Y::LPR;
    const uint32_t t = tensor_rows<THREADS>(S, tcols);
#pragma unroll 2
    for (int st = 0; st < R.tsteps; ++st) {
        const int i = i0 + st * STEP;
        float4 v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            v[c] = i < R.nt ? __ldcg(reinterpret_cast<const float4 *>(R.g + (size_t)(R.ns + i) * RP) + c * Y::LPR + cl) : make_float4(0.f, 0.f, 0.f, 0.f);
        tensor_store16(t + st * CPL, v);
    }
    sm100::tmem_wait_st();
}

template <int RP, int CPL, int THREADS>
__device__ __forceinline__ Lane<RP, CPL> make_lane(const Shared &S, int tcols)
{
    typedef Lay<RP, CPL> Y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Lane<RP, CPL> L;
    L.t = tcols ? tensor_rows<THREADS>(S, tcols) : 0;
    L.cl = lane % Y::LPR;
    L.i0 = warp * Y::RPW + lane / Y::LPR;
#pragma unroll
    for (int v = 0; v < Y::NV; ++v) L.k[v] = smem_addr(S.K) + (L.i0 * Y::CH + Y::swz(L.i0, v * Y::LPR + L.cl)) * 16;
    L.w = smem_addr(S.w) + L.cl * 16;
    // after the halving the lane holds its columns off .. off + LEFT - 1 (warp_columns)
    int off = 0;
#pragma unroll
    for (int bit = Y::LPR, h = CPL / 2; bit < 32; bit <<= 1, h >>= 1) off += (lane & bit) ? h : 0;
    L.red = smem_addr(S.work) + (warp * RP + ((off >> 2) * Y::LPR + L.cl) * 4 + (off & 3)) * 4;
    L.own = smem_addr(S.work) + threadIdx.x * 4;
    return L;
}

// One pass over the block's rows: the lane's column sums.  CLOSE: the reciprocal row sums go to inv_out instead (0 for a
// token without weight).  WEIGHTED: the tokens bring weights of their own.
template <int RP, int CPL, int THREADS, bool TENSOR, bool CLOSE, bool WEIGHTED>
__device__ __forceinline__ void pass_t(const Lane<RP, CPL> &L, const Share &R, const u64 (&w)[CPL / 2], u64 (&acc)[CPL / 2], float *inv_out)
{
    typedef Lay<RP, CPL> Y;
    constexpr int STEP = (THREADS / 32) * Y::RPW;        // a multiple of 8: a lane's chunk permutation never changes
#pragma unroll
    for (int j = 0; j < CPL / 2; ++j) acc[j] = 0;
    auto one = [&](const Row<CPL> &k, int i, int end) {
        float m = 1.f;
        if (WEIGHTED) m = i < end ? __ldg(R.mass + i) : 0.f;
        if (!CLOSE) {
            row_step<RP, CPL, true>(k, w, acc, m);
        } else {
            const float inv = row_step<RP, CPL, false>(k, w, acc, 1.f);
            if (i < end && L.cl == 0) inv_out[i] = m > 0.f ? inv : 0.f;
        }
    };
    auto load = [&](Row<CPL> &k, int st) {
#pragma unroll
        for (int v = 0; v < Y::NV; ++v) lds2(k.k[2 * v], k.k[2 * v + 1], L.template chunk<TENSOR && RP <= 32>(st * (STEP * RP * 4), v));
    };
    auto fetch = [&](Row<CPL> (&k)[2], int i) {              // two steps' rows from L2
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int v = 0; v < Y::NV; ++v) {
                const ulonglong2 t = i + u * STEP < R.nrows
                                         ? __ldcg(reinterpret_cast<const ulonglong2 *>(R.g + (size_t)(i + u * STEP) * RP) + v * Y::LPR + L.cl)
                                         : make_ulonglong2(0, 0);
                k[u].k[2 * v] = t.x;
                k[u].k[2 * v + 1] = t.y;
            }
    };
    if constexpr (!TENSOR) {
        if (R.steps & 1) {
            Row<CPL> k;
            load(k, 0);
            one(k, L.i0, R.ns);
        }
        for (int st = R.steps & 1; st < R.steps; st += 2) {
            Row<CPL> k[2];
            load(k[0], st);
            load(k[1], st + 1);
            one(k[0], L.i0 + st * STEP, R.ns);
            one(k[1], L.i0 + (st + 1) * STEP, R.ns);
        }
        if (R.ns < R.nrows)                                  // rows that do not fit: streamed from L2
            for (int i = R.ns + L.i0; i - L.i0 < R.nrows; i += 2 * STEP) {
                Row<CPL> k[2];
                fetch(k, i);
#pragma unroll
                for (int u = 0; u < 2; ++u) one(k[u], i + u * STEP, R.nrows);
            }
    } else {
        int st = R.steps & 1;
        if (st) {
            Row<CPL> k;
            load(k, 0);
            one(k, L.i0, R.ns);
        }
        auto shared_pair = [&]() {
            Row<CPL> k[2];
            load(k[0], st);
            load(k[1], st + 1);
            one(k[0], L.i0 + st * STEP, R.ns);
            one(k[1], L.i0 + (st + 1) * STEP, R.ns);
            st += 2;
        };
        // rows that fit neither place, requested in front of a pair of steps from shared memory
        const int on_chip = R.ns + R.nt;
        if (on_chip < R.nrows)
            for (int i = on_chip + L.i0; i - L.i0 < R.nrows; i += 2 * STEP) {
                Row<CPL> k[2];
                fetch(k, i);
                if (st < R.steps) shared_pair();
#pragma unroll
                for (int u = 0; u < 2; ++u) one(k[u], i + u * STEP, R.nrows);
            }
        // tensor memory, likewise
#pragma unroll 1
        for (int ts = 0; ts < R.tsteps; ts += 2) {
            u64 k2[CPL];
            tensor_load<2 * CPL>(k2, L.t + ts * CPL);
            if (st < R.steps) shared_pair();
            tensor_settle<2 * CPL>(k2);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                Row<CPL> k;
#pragma unroll
                for (int j = 0; j < CPL / 2; ++j) k.k[j] = k2[u * (CPL / 2) + j];
                one(k, R.ns + L.i0 + (ts + u) * STEP, on_chip);
            }
        }
        while (st < R.steps) shared_pair();
    }
}

template <int RP, int CPL, int THREADS, bool TENSOR, bool CLOSE>
__device__ __forceinline__ void pass(const Lane<RP, CPL> &L, const Share &R, const u64 (&w)[CPL / 2], u64 (&acc)[CPL / 2], float *inv_out)
{
    if (R.mass == nullptr) pass_t<RP, CPL, THREADS, TENSOR, CLOSE, false>(L, R, w, acc, inv_out);
    else pass_t<RP, CPL, THREADS, TENSOR, CLOSE, true>(L, R, w, acc, inv_out);
}

template <int RP, int CPL>
__device__ __forceinline__ void load_weights(const Lane<RP, CPL> &L, u64 (&w)[CPL / 2])
{
#pragma unroll
    for (int v = 0; v < CPL / 4; ++v) lds2(w[2 * v], w[2 * v + 1], L.w + v * (Lay<RP, CPL>::LPR * 16));
}

template <int CNT, int N, int BIT, bool MAX>
__device__ __forceinline__ void halve_lanes(float (&v)[N], int lane, int &off)
{
    if constexpr (BIT < 32) {
        constexpr int H = CNT > 1 ? CNT / 2 : 1;
        const bool up = CNT > 1 && (lane & BIT) != 0;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const float give = up || CNT == 1 ? v[i] : v[i + H < N ? i + H : i], keep = up ? v[i + H < N ? i + H : i] : v[i];
            const float got = __shfl_xor_sync(0xffffffffu, give, BIT);
            v[i] = MAX ? fmaxf(keep, got) : keep + got;
        }
        off += up ? H : 0;
        halve_lanes<H, N, BIT * 2, MAX>(v, lane, off);
    }
}

// The warp's column values into red[warp][RP], in a fixed order: lanes that hold the same columns halve them among them.
template <int RP, int CPL, bool MAX>
__device__ __forceinline__ void warp_columns(float *red, float (&v)[CPL])
{
    typedef Lay<RP, CPL> Y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cl = lane % Y::LPR;
    int off = 0;
    halve_lanes<CPL, CPL, Y::LPR, MAX>(v, lane, off);
    constexpr int LEFT = CPL / Y::RPW < 1 ? 1 : CPL / Y::RPW;
#pragma unroll
    for (int i = 0; i < LEFT; ++i) {
        const int k = off + i;
        red[warp * RP + ((k >> 2) * Y::LPR + cl) * 4 + (k & 3)] = v[i];
    }
}

// ... and the block's: thread t < RP returns column t's.  One barrier inside; the work area is free again after the
// caller's next barrier.
template <int RP, int CPL, int THREADS, bool MAX>
__device__ __forceinline__ float block_columns(const Shared &S, float (&v)[CPL])
{
    float *red = reinterpret_cast<float *>(S.work);
    warp_columns<RP, CPL, MAX>(red, v);
    __syncthreads();
    float tot = MAX ? neg_inf() : 0.f;
    if (threadIdx.x < RP) {
#pragma unroll
        for (int wv = 0; wv < THREADS / 32; ++wv) {
            const float o = red[wv * RP + threadIdx.x];
            tot = MAX ? fmaxf(tot, o) : tot + o;
        }
    }
    return tot;
}

// ---------------------------------------------------------------------------------------------------------------
// The exchange between the blocks of a group
// ---------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void put_word(u64 *p, float v, unsigned tag)
{
    const u64 word = ((u64)tag << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(word) : "memory");
}
__device__ __forceinline__ u64 peek_word(const u64 *p)
{
    u64 v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t in_peer(uint32_t addr, int block)
{
    uint32_t o;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(addr), "r"(block));
    return o;
}
// A float into another block's shared memory, counted by that block's barrier.
__device__ __forceinline__ void send(uint32_t dst, float v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst), "r"(__float_as_uint(v)), "r"(bar)
                 : "memory");
}
// Whether the bytes of a set of sends have arrived.
__device__ __forceinline__ bool sends_arrived(uint32_t bar, unsigned parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Wait for them (at most a second, then the call is flagged and every later wait gives up at once); false if they did not come.
__device__ __forceinline__ bool wait_sends(uint32_t bar, unsigned parity, volatile int *dead, int *status)
{
    u64 start = 0;
    for (unsigned spin = 1;; ++spin) {
        if (sends_arrived(bar, parity)) return true;
        if ((spin & 63u) != 0) continue;
        const u64 now = global_timer_ns();
        if (start == 0) start = now;
        if (*dead || now - start > kWaitNs) {
            if (!*dead) atomicOr(status, 4 /* LOT_DEV_TIMEOUT */);
            *dead = 1;
            return false;
        }
    }
}

// Bytes of shared memory in which a block of a cluster receives, two sets; the barriers that count them are behind the flags.
__host__ __device__ constexpr int peer_bytes(int RP, int C, int K) { return K == 1 ? 0 : 2 * RP * 4 * (C == K ? C : 1); }

// Before the first exchange of a launch, and behind the last (nobody's shared memory is written any more).
template <int RP, typename Args>
__device__ __forceinline__ void open_exchange(const Args &a, const Shared &S)
{
    if (a.K == 1) return;
    if (threadIdx.x == 0) {
        for (int b = 0; b < 2; ++b) {
            sm100::mbar_init(S.bars + 8 * b, 1);
            sm100::mbar_arrive_expect_tx(S.bars + 8 * b, peer_bytes(RP, a.C, a.K) / 2);
        }
        sm100::fence_barrier_init();
    }
    __syncthreads();
    cluster_sync();
}
template <typename Args> __device__ __forceinline__ void close_exchange(const Args &a)
{
    if (a.K > 1) cluster_sync();
}

// The block's tensor memory, before its first use (the block waits behind it) and behind the last.
__device__ __forceinline__ void open_tensor(const Shared &S, int tcols)
{
    if (tcols == 0) return;
    if (threadIdx.x < 32) {
        sm100::tmem_alloc(S.tmem, tcols);
        sm100::tmem_relinquish();
    }
    sm100::tc_fence_before();
    __syncthreads();
    sm100::tc_fence_after();
}
__device__ __forceinline__ void close_tensor(const Shared &S, int tcols)
{
    if (tcols == 0) return;
    sm100::tc_fence_before();
    __syncthreads();
    sm100::tc_fence_after();
    if (threadIdx.x < 32) {
        uint32_t base;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(base) : "r"(S.tmem) : "memory");
        sm100::tmem_dealloc(base, tcols);
    }
}

// Totals of the group's column values, the same bits in every block: thread t < RP gives its block's value of column t and
// gets the group's.  The group's C blocks are M = C / K clusters of K.
//   M = 1: every block sends its values into all others' shared memory.
//   else:  the blocks of a cluster first add up RP / K columns each (sent as above), and leave the sums of the cluster
//          as words in the L2, of which every block reads M a column.
// What this costs is latency, a trip through the cluster's shared memory (0.5 us) and one through L2 (0.6); every wait is for
// all words of a thread at once.  A loop of nothing but exchanges, at RP = 256: clusters of eight 1.07 us at 24 blocks, 1.13 at
// 48, 1.47 at 72; of two 1.06 at 8, 1.6 at 24, 2.2 at 48, 3.1 at 72; with every block's words read by every block up to 16
// blocks and columns owned by blocks above, both through L2, it was 2.0 at 8, 4.6 at 24, 5.4 at 48, 5.9 at 72.
// Two sets of everything by parity: a block can be at most one exchange ahead of the others.
template <int RP, int THREADS, bool MAX, typename Args>
__device__ __forceinline__ float group_columns(const Args &a, const Shared &S, float part, int group, int c, unsigned &seq)
{
    const int C = a.C, K = a.K, tid = threadIdx.x;
    if (C == 1) return part;
    // A thread whose wait gave up (the call is flagged, its results are void) sends, waits for and arms nothing any more, and with its columns missing
    // the threads that need them give up in turn: no barrier is armed whose phase is still open (its count would be undefined), and none
    // counts more bytes than a few exchanges bring.  Each thread goes by its own waits: with a flag of the block read in every exchange B = 4,
    // H = 8, n = 16384, d = 128, r = 128, T = 20 took 1680 us, now 1669, and n = 4096, H = 16, r = 64 (read in front of the sends) 65.4, 64.2.
    constexpr unsigned kGaveUp = ~0u;
    if (seq == kGaveUp) return part;
    const unsigned nth = seq - a.seq0;                       // of this launch
    ++seq;
    const unsigned tag = seq;
    auto join = [](float x, float y) { return MAX ? fmaxf(x, y) : x + y; };
    const float none = MAX ? neg_inf() : 0.f;
    const uint32_t bar = S.bars + 8 * (nth & 1), mine = S.peers + (nth & 1) * (peer_bytes(RP, C, K) / 2);
    const unsigned parity = (nth >> 1) & 1;
    auto add_up = [&](int stride) {                          // the values of K blocks, `stride` floats apart
        float v[8];
#pragma unroll
        for (int o = 0; o < 8; ++o) v[o] = o < K ? lds(mine + (o * stride + tid) * 4) : none;
#pragma unroll
        for (int h = 4; h > 0; h >>= 1)
#pragma unroll
            for (int o = 0; o < h; ++o) v[o] = join(v[o], v[o + h]);
        return v[0];
    };
    if (C == K) {
        if (tid < RP) {
            for (int o = 0; o < K; ++o) send(in_peer(mine + (c * RP + tid) * 4, o), part, in_peer(bar, o));
            const bool all = wait_sends(bar, parity, S.flag, a.status);
            part = add_up(RP);
            if (tid == 0 && all) sm100::mbar_arrive_expect_tx(bar, peer_bytes(RP, C, K) / 2);      // for the exchange after the next
            if (!all) seq = kGaveUp;
        }
        return part;
    }
    const int M = C / K, m = c / K, rank = c % K;
    u64 *X = a.xbuf + (size_t)(group * 2 + (seq & 1)) * M * RP;
    if (K == 1) {
        if (tid < RP) put_word(X + (size_t)c * RP + tid, part, tag);
    } else {
        const int own = RP / K, sh = 31 - __clz(own);
        if (tid < RP) {
            const int to = tid >> sh;
            send(in_peer(mine + (rank * own + (tid & (own - 1))) * 4, to), part, in_peer(bar, to));
        }
        if (tid < own) {
            const bool all = wait_sends(bar, parity, S.flag, a.status);
            if (all) put_word(X + (size_t)m * RP + rank * own + tid, add_up(own), tag);
            if (tid == 0 && all) sm100::mbar_arrive_expect_tx(bar, peer_bytes(RP, C, K) / 2);
        }
    }
    float tot = none;
    bool dead = false;
    if (tid < RP)
        for (int m0 = 0; m0 < M; m0 += kWords) {
            const u64 *p = X + (size_t)m0 * RP + tid;
            u64 wd[kWords], start = 0;
#pragma unroll
            for (int u = 0; u < kWords; ++u) wd[u] = m0 + u < M ? peek_word(p + u * RP) : (u64)tag << 32 | __float_as_uint(none);
            for (unsigned spin = 1;; ++spin) {
                bool all = true;
#pragma unroll
                for (int u = 0; u < kWords; ++u)
                    if ((unsigned)(wd[u] >> 32) != tag) {
                        wd[u] = peek_word(p + u * RP);
                        all = false;
                    }
                if (all) break;
                if ((spin & 63u) != 0) continue;
                const u64 now = global_timer_ns();
                if (start == 0) start = now;
                if (*S.flag || now - start > kWaitNs) {
                    if (!*S.flag) atomicOr(a.status, 4 /* LOT_DEV_TIMEOUT */);
                    *S.flag = 1;
                    dead = true;
                    break;
                }
            }
#pragma unroll
            for (int u = 0; u < kWords; ++u) tot = join(tot, __uint_as_float((unsigned)wd[u]));
        }
    if (dead) seq = kGaveUp;
    return tot;
}

// Column sums in the log domain, from stored exponents e_it: with x_it = e_it - log2 sum_t 2^e_it + log2 m_i the
// thread t < RP returns log2 sum_i 2^x_it over the group, taken relative to the column's maximum.
template <int RP, int CPL, int THREADS>
__device__ __forceinline__ float log_columns(const SweepArgs &a, const Shared &S, const Share &R, int group, int c, unsigned &seq)
{
    typedef Lay<RP, CPL> Y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane / Y::LPR, cl = lane % Y::LPR;
    constexpr int STEP = (THREADS / 32) * Y::RPW;
    float v[CPL];
#pragma unroll
    for (int k = 0; k < CPL; ++k) v[k] = neg_inf();
    for (int base = warp * Y::RPW; base < R.nrows; base += STEP) {
        const int i = base + sub;
        const bool ok = i < R.nrows;
        float e[CPL];
        float s = 0.f;
#pragma unroll
        for (int u = 0; u < Y::NV; ++u) {
            const float4 t = ok ? *chunk_ptr<RP, CPL>(S, R, i, u * Y::LPR + cl) : make_float4(0.f, 0.f, 0.f, 0.f);
            e[4 * u] = t.x; e[4 * u + 1] = t.y; e[4 * u + 2] = t.z; e[4 * u + 3] = t.w;
        }
#pragma unroll
        for (int k = 0; k < CPL; ++k) s += ex2(e[k]);
        s = group_sum(s, Y::LPR);
        const float m = ok ? (R.mass ? __ldg(R.mass + i) : 1.f) : 0.f;
        const float shift = m > 0.f ? lg2(m) - lg2(s) : neg_inf();
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            e[k] = e[k] + shift;
            v[k] = fmaxf(v[k], e[k]);
        }
        if (ok) {
#pragma unroll
            for (int u = 0; u < Y::NV; ++u)
                *chunk_ptr<RP, CPL>(S, R, i, u * Y::LPR + cl) = make_float4(e[4 * u], e[4 * u + 1], e[4 * u + 2], e[4 * u + 3]);
        }
    }
    const float kap = group_columns<RP, THREADS, true>(a, S, block_columns<RP, CPL, THREADS, true>(S, v), group, c, seq);
    if (threadIdx.x < RP) S.w[threadIdx.x] = kap;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < CPL; ++k) v[k] = 0.f;
    for (int base = warp * Y::RPW; base < R.nrows; base += STEP) {
        const int i = base + sub;
        if (i >= R.nrows) continue;
#pragma unroll
        for (int u = 0; u < Y::NV; ++u) {
            const float4 t = *chunk_ptr<RP, CPL>(S, R, i, u * Y::LPR + cl), kk = *reinterpret_cast<const float4 *>(S.w + (u * Y::LPR + cl) * 4);
            if (kk.x > neg_inf()) v[4 * u] += ex2(t.x - kk.x);
            if (kk.y > neg_inf()) v[4 * u + 1] += ex2(t.y - kk.y);
            if (kk.z > neg_inf()) v[4 * u + 2] += ex2(t.z - kk.z);
            if (kk.w > neg_inf()) v[4 * u + 3] += ex2(t.w - kk.w);
        }
    }
    __syncthreads();
    const float sum = group_columns<RP, THREADS, false>(a, S, block_columns<RP, CPL, THREADS, false>(S, v), group, c, seq);
    return kap + lg2(sum);
}

// The group's share of problem p for block c, and the block's shared memory.
template <typename T, int RP, int THREADS>
__device__ __forceinline__ Shared carve(uint8_t *p, int srows, size_t work = work_bytes<T>(RP, THREADS), size_t ref = ref_bytes(RP, THREADS))
{
    Shared S;
    S.K = reinterpret_cast<float *>(p); p += (size_t)srows * RP * 4;
    S.gref = reinterpret_cast<double *>(p); p += RP * 8;
    S.work = p; p += work;
    S.ref = reinterpret_cast<float *>(p); p += ref;
    S.w = reinterpret_cast<float *>(p); p += RP * 4;
    S.tgt = reinterpret_cast<float *>(p); p += RP * 4;
    S.flag = reinterpret_cast<volatile int *>(p);
    S.bars = smem_addr(p) + 16;
    S.peers = smem_addr(p) + 64;
    S.tmem = smem_addr(p) + 32;
    return S;
}

struct Problem {
    int slice, side, h, n, nv, row0;
};

template <int RP, int CPL, int THREADS>
__device__ __forceinline__ Problem locate(const SweepArgs &a, int p, int c, Share &R)
{
    constexpr int STEP = (THREADS / 32) * Lay<RP, CPL>::RPW;
    Problem P;
    const int BH = a.B * a.H;
    P.slice = p >> 1;
    P.side = (p & 1) ^ 1;
    if (a.n[0] != a.n[1]) {                                  // the longer side's problems first: groups then share both evenly
        P.slice = p < BH ? p : p - BH;
        P.side = (p < BH) == (a.n[1] > a.n[0]);
    }
    P.h = P.slice % a.H;
    P.n = a.n[P.side];
    P.nv = P.n;
    if (P.side == 1 && a.key_len != nullptr) P.nv = min(max(__ldg(a.key_len + P.slice / a.H), 0), P.n);
    P.nv = max(P.nv - a.skip, 0);
    const int per = (P.nv + a.C - 1) / a.C;
    P.row0 = min(c * per, P.nv);
    R.nrows = min(per, P.nv - P.row0);
    P.row0 += a.skip;                                        // from here on within the slice's tokens
    R.ns = min(R.nrows, a.srows);
    R.steps = (R.ns + STEP - 1) / STEP;
    R.nt = min(R.nrows - R.ns, a.tcols / lane_sharers(THREADS) / CPL * STEP);
    R.tsteps = (R.nt + 2 * STEP - 1) / (2 * STEP) * 2;
    R.g = a.kt[P.side] ? a.kt[P.side] + ((size_t)P.slice * P.n + P.row0) * RP : nullptr;
    R.mass = a.mass[P.side] ? a.mass[P.side] + (size_t)P.slice * P.n + P.row0 : nullptr;
    return P;
}

// The block's rows from global into shared memory; rows up to the next full step are filled with zeros.  The caller waits
// for the copies (cp.async.wait_group 0) and then for the block.
template <int RP, int CPL, int THREADS>
__device__ __forceinline__ void load_rows(const Shared &S, const Share &R)
{
    constexpr int STEP = (THREADS / 32) * Lay<RP, CPL>::RPW;
    for (int idx = threadIdx.x; idx < R.steps * STEP * (RP / 4); idx += THREADS) {
        const int i = idx / (RP / 4);
        const uint32_t dst = smem_addr(reinterpret_cast<float4 *>(S.K + (size_t)i * RP) + Lay<RP, CPL>::swz(i, idx % (RP / 4)));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(reinterpret_cast<const float4 *>(R.g) + (i < R.ns ? idx : 0)),
                     "r"(i < R.ns ? 16 : 0) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Whether a weight is outside the kernel's range, and whether that is because its column sum (target / weight) left
// float32's.
__device__ __forceinline__ bool out_of_range(float w) { return !(w >= kFarLo && w <= kFarHi); }
__device__ __forceinline__ bool sum_lost(float tgt, float w) { return !(tgt >= kLostLo * w && tgt <= kLostHi * w); }

// One iteration of the block's problem: thread t < r gets its column's weight before and after; true where the update
// leaves the range (block-uniform; the weights in shared memory are then the new ones all the same).  The chain of an
// iteration is what a short problem takes: two plain barriers, the range flag read beside the weights of the next
// iteration (a voting barrier took 50 cycles more).
template <int RP, int CPL, int THREADS, bool GROUP, bool TENSOR>
__device__ __forceinline__ bool iterate(const SweepArgs &a, const Shared &S, const Share &R, const Lane<RP, CPL> &L, u64 (&w)[CPL / 2],
                                        float tgt, int group, int c, unsigned &seq, float &wold, float &wnew)
{
    typedef Lay<RP, CPL> Y;
    u64 acc[CPL / 2];
    pass<RP, CPL, THREADS, TENSOR, false>(L, R, w, acc, nullptr);
    float v[CPL];
#pragma unroll
    for (int j = 0; j < CPL / 2; ++j) unpack_f2(acc[j], v[2 * j], v[2 * j + 1]);
    int off = 0;
    halve_lanes<CPL, CPL, Y::LPR, false>(v, threadIdx.x & 31, off);
    constexpr int LEFT = CPL / Y::RPW < 1 ? 1 : CPL / Y::RPW;
#pragma unroll
    for (int i = 0; i < LEFT; ++i) sts(L.red + ((i >> 2) * Y::LPR * 4 + (i & 3)) * 4, v[i]);
    __syncthreads();
    float tot = 0.f;
    if (threadIdx.x < RP) {
        if (TENSOR) { tgt = S.tgt[threadIdx.x]; wnew = S.w[threadIdx.x]; }       // not kept over the pass: three registers
        float o[THREADS / 32];
#pragma unroll
        for (int i = 0; i < THREADS / 32; ++i) o[i] = lds(L.own + i * (RP * 4));
#pragma unroll
        for (int h = THREADS / 64; h > 0; h >>= 1)
#pragma unroll
            for (int i = 0; i < h; ++i) o[i] += o[i + h];
        tot = o[0];
    }
    if (GROUP) tot = group_columns<RP, THREADS, false>(a, S, tot, group, c, seq);
    if ((int)threadIdx.x < a.r) {
        wold = wnew;
        wnew = tgt * rcp(tot);
        if (out_of_range(wnew)) S.flag[1] = 1;
        S.w[threadIdx.x] = wnew;
    }
    __syncthreads();
    load_weights<RP, CPL>(L, w);
    return S.flag[1] != 0;
}

// The rest of a problem's iterations from `it` on, whose update left the kernel's range (wold, wnew: thread t < r's weight
// before and after it): the kernel is rebuilt around the new potentials, after the update has been redone in the log
// domain where a column sum was lost.  Out of line and behind the iteration loop, so that it costs the loop no registers.  Returns the sequence number.
template <typename T, int RP, int CPL, int THREADS, bool GROUP, bool TENSOR, size_t WORK = work_bytes<T>(RP, THREADS), size_t REF = ref_bytes(RP, THREADS)>
__device__ __noinline__ unsigned recover(const SweepArgs *ap, int p, int group, int c, int it, unsigned seq, float wold, float wnew)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const SweepArgs &a = *ap;
    const Shared S = carve<T, RP, THREADS>(smem, a.srows, WORK, REF);
    Share R;
    const Problem P = locate<RP, CPL, THREADS>(a, p, c, R);
    const T *x = static_cast<const T *>(a.x[P.side]) + ((size_t)P.slice * P.n + P.row0) * a.d;
    const float *z = a.z + (size_t)P.h * a.r * a.d;
    const Lane<RP, CPL> L = make_lane<RP, CPL, THREADS>(S, a.tcols);
    const int tid = threadIdx.x, r = a.r, NP = 2 * a.B * a.H;
    // the kept potentials of every iteration (backward): as they are, and at the end relative to the last kernel
    const bool keep = a.hist != nullptr && c == 0 && tid < r;
    double *hg = a.hist_g + (size_t)p * RP + tid;
    if (keep)
        for (int k = 0; k <= it; ++k) hg[(size_t)k * NP * RP] = S.gref[tid] + log2((double)a.hist[((size_t)k * NP + p) * RP + tid]);
    while (true) {
        double gn = 0.0;
        if (__syncthreads_or(tid < r && sum_lost(S.tgt[tid < RP ? tid : 0], wnew))) {
            if (tid < r) {
                gn = S.gref[tid] + log2((double)wold);
                S.gref[tid] = gn;
            }
            __syncthreads();
            build<T, RP, CPL, THREADS, true>(S, R, x, z, a.d, r, a.scale);
            const float lam = log_columns<RP, CPL, THREADS>(a, S, R, group, c, seq);
            if (tid < r) gn += log2((double)S.tgt[tid]) - (double)lam;
        } else if (tid < r) {
            gn = S.gref[tid] + log2((double)wnew);
        }
        __syncthreads();
        if (tid < r) {
            if (!isfinite(gn)) atomicOr(a.status, 1 /* LOT_DEV_NONFINITE */);
            if (keep) hg[(size_t)(it + 1) * NP * RP] = gn;
            S.gref[tid] = gn - (double)kStartLog2;
            S.w[tid] = kStart;
        } else if (tid < RP) {
            S.w[tid] = 0.f;
        }
        if (tid == 0) S.flag[1] = 0;
        __syncthreads();
        build<T, RP, CPL, THREADS, false>(S, R, x, z, a.d, r, a.scale);
        if constexpr (TENSOR) load_tensor_rows<RP, CPL, THREADS>(S, R, a.tcols);
        bool bad = false;
        u64 w[CPL / 2];
        load_weights<RP, CPL>(L, w);
        wnew = kStart;
        for (++it; it < a.iters && !bad; ++it) {
            bad = iterate<RP, CPL, THREADS, GROUP, TENSOR>(a, S, R, L, w, S.tgt[tid < RP ? tid : 0], group, c, seq, wold, wnew);
            if (keep && !bad) hg[(size_t)(it + 1) * NP * RP] = S.gref[tid] + log2((double)wnew);
        }
        if (!bad) break;
        --it;                                                // the iteration whose update has to be redone
    }
    if (a.hist != nullptr && c == 0) {
        bool wide = false;
        for (int k = 0; tid < RP && k <= a.iters; ++k) {
            const float v = tid < r ? (float)exp2(hg[(size_t)k * NP * RP] - S.gref[tid]) : 0.f;
            wide = wide || (tid < r && !(v >= kHistLo && v <= kHistHi));
            a.hist[((size_t)k * NP + p) * RP + tid] = v;
        }
        wide = __syncthreads_or(wide);
        if (tid == 0) a.wide[p] = wide;
    }
    return seq;
}

} // namespace sweep
} // namespace lot
