// Long sequences with 16 < r <= 64 pivots (bf16 tensors, d = 64): the Gibbs kernel as bf16, built and iterated on in one
// launch, then applied by the tensor-core kernels of lot_apply.cu.
//
// As in lot_sweep.cu a problem (one side of one slice) is shared by a group of C blocks and every pass is two
// multiply-adds per entry on the stored kernel, here K_it = 2^(L_it + Gref_t - ref_i) <= 2^67 in bf16 (the rounding the
// streamed path has always had; potentials to about 1e-4): half the bytes, so a pass over n = 16384, H = 16 reads 67 MB, of
// which the blocks keep the first rows of their share in shared memory and the rest comes from L2.  Each block
// computes the logits of its own rows (warp-level products, Z as bf16 hi + lo), so building one group's kernel
// overlaps another's passes.  At n = 4096, H = 16, r = 64, T = 10: 42 us (17 of them building) of a call of 64, which took 117 on
// the streamed path; at n = 16384 132 (52) of 171, against 190 (47 of 71 and 135 of 180 with the exchanges polled in L2).  A pass is bound by latency: per
// scheduler four warps, whose registers hold the weights, the column sums and two rows, issue in 40% of the cycles.
//
// The key side is applied from twice bf16's precision, as the streamed path's apply passes do with recomputed logits: the
// building also leaves K minus its rounding, which only apply_w reads (1.4 us of a call at n = 4096; 12 at n = 16384: 34 MB
// written, 6 us, read again, 5, and in the L2 in place of other rows).  When all problems together exceed the L2, groups are
// made larger and work through the problems in rounds, so that what is iterated on stays in the L2.
#include "lot_chain.cuh"
#include "lot_sweep_core.cuh"

namespace lot {
namespace stream {

using namespace sweep;

constexpr int kThreads = 256, kD = 64, RP = 64;
constexpr int kRowsStep = 64;              // rows per step of a block: eight a warp, four lanes a row
constexpr int kZPitch = 144;               // bytes per staged pivot row (conflict-free ldmatrix)
constexpr int kStage = 2 * RP * kZPitch;   // staged pivots (hi, lo): in the kernel rows' area while building
constexpr int kWork = kThreads / 32 * RP * 4;
constexpr int kFixed = kWork + kThreads * 4 + RP * 20 + 64 + 2 * kPeers * RP * 4;

constexpr int kRowsCap = (kSmemPerSM / 2 - kSmPerBlockReserve - kFixed) / 128 / kRowsStep * kRowsStep;       // kernel rows a block has room for, two blocks an SM
constexpr int kMostWords = 80;             // words a column that a thread reads, sixteen at a time

__host__ __device__ constexpr int area_bytes(int srows) { return srows * 128 > kStage ? srows * 128 : kStage; }

struct StreamArgs {
    const __nv_bfloat16 *x[2];
    const float *z, *beta;
    const int32_t *key_len;
    uint8_t *kt;               // [2][BH][npad][64] bf16, side 0 queries
    uint8_t *low;              // [BH][n][64] bf16: the key side's kernel minus its bf16 rounding, or nullptr
    float *G;                  // [2][BH][64] log2 of the final weights (relative to the kernel as stored)
    int *decision;             // [2][BH], set to 1
    float *g_out[2];
    u64 *xbuf;
    int *status;
    int B, H, n, npad, r, T, C, K, groups, srows;
    unsigned seq0;             // 0
    double scale, eps_ln2;
};

struct Mem {
    uint8_t *K, *z;            // [srows][128 bytes]; its last bytes hold the pivots while building
    float *before;             // the weights before the last update
    Shared s;
};

__device__ __forceinline__ Mem carve16(uint8_t *p, int srows)
{
    Mem m;
    m.K = p; p += area_bytes(srows);
    m.z = p - kStage;
    m.s.K = nullptr;
    m.s.gref = reinterpret_cast<double *>(p); p += RP * 8;
    m.s.work = p; p += kWork;
    m.s.ref = reinterpret_cast<float *>(p); p += kThreads * 4;
    m.s.w = reinterpret_cast<float *>(p); p += RP * 4;
    m.s.tgt = reinterpret_cast<float *>(p); p += RP * 4;
    m.before = reinterpret_cast<float *>(p); p += RP * 4;
    m.s.flag = reinterpret_cast<volatile int *>(p);    // [0], [1] as in the sweep kernels; [2], [3]: see solve16
    m.s.bars = smem_addr(p) + 16;
    m.s.peers = smem_addr(p) + 64;
    return m;
}

struct Part {                  // a block's share of a problem
    int slice, side, h, nv, row0, nrows, ns, steps;
    uint8_t *g, *low;          // its rows in global memory, and those of the low half or nullptr
    const __nv_bfloat16 *x;
};

__device__ __forceinline__ Part locate16(const StreamArgs &a, int p, int c)
{
    Part P;
    P.slice = p >> 1;
    P.side = (p & 1) ^ 1;
    P.h = P.slice % a.H;
    P.nv = a.n;
    if (P.side == 1 && a.key_len != nullptr) P.nv = min(max(__ldg(a.key_len + P.slice / a.H), 0), a.n);
    const int per = (P.nv + a.C - 1) / a.C;
    P.row0 = min(c * per, P.nv);
    P.nrows = min(per, P.nv - P.row0);
    P.ns = min(P.nrows, a.srows);
    P.steps = (P.ns + kRowsStep - 1) / kRowsStep;
    P.g = a.kt + ((size_t)(P.side * a.B * a.H + P.slice) * a.npad + P.row0) * 128;
    P.low = P.side == 1 && a.low != nullptr ? a.low + ((size_t)P.slice * a.n + P.row0) * 128 : nullptr;
    P.x = a.x[P.side] + ((size_t)P.slice * a.n + P.row0) * kD;
    return P;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&t);
}

// The order of the products' operands is free as long as both sides agree.  A lane's token values of two steps are eight
// neighbours in memory, and its eight results of four tiles are eight neighbouring pivots: 16-byte loads and stores, a
// quarter of the requests of the instruction's own layout (whose 4-byte loads and 8-byte stores held the load-store
// unit for most of the 72 us that building took at n = 16384, H = 16).
__device__ __forceinline__ int pivot_of(int j, int q, int e) { return 32 * (j >> 2) + 8 * q + 2 * (j & 3) + e; }

// Pivots of the head in base-2 logit units as bf16 hi + lo.
__device__ __forceinline__ void stage_pivots(const StreamArgs &a, const Mem &m, const Part &P)
{
    const float *z = a.z + (size_t)P.h * a.r * kD;
    const float scale = (float)a.scale;
    float2 zz[RP * kD / 2 / kThreads];
#pragma unroll
    for (int u = 0; u < RP * kD / 2 / kThreads; ++u) {
        const int idx = threadIdx.x + u * kThreads, t = idx / (kD / 2);
        zz[u] = t < a.r ? __ldg(reinterpret_cast<const float2 *>(z + (size_t)t * kD + (idx % (kD / 2)) * 2)) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < RP * kD / 2 / kThreads; ++u) {
        const int idx = threadIdx.x + u * kThreads, t = idx / (kD / 2), c = (idx % (kD / 2)) * 2;
        const int row = (t & 32) | (t & 6) << 2 | (t >> 2 & 6) | (t & 1);                     // pivot_of(row / 8, ...) = t
        const int col = (c & 32) | (c & 4) << 2 | (c & 2) << 2 | (c >> 2 & 6);                // as fetch_tokens
        const float x0 = zz[u].x * scale, x1 = zz[u].y * scale;
        const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
        *reinterpret_cast<__nv_bfloat162 *>(m.z + row * kZPitch + col * 2) = h;
        *reinterpret_cast<uint32_t *>(m.z + (RP + row) * kZPitch + col * 2) = pack2(x0 - __low2float(h), x1 - __high2float(h));
    }
    __syncthreads();
}

// Logits of 16 rows a warp, all pivots: tokens straight from global memory, pivots from shared memory.
__device__ __forceinline__ void fetch_tokens(uint32_t (&a)[kD / 16][4], const Part &P, int rt)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int kk = 0; kk < kD / 32; ++kk) {
            const int i = rt + warp * 16 + g + e * 8;
            const uint4 v = i < P.nrows ? __ldg(reinterpret_cast<const uint4 *>(P.x + (size_t)i * kD + kk * 32 + 8 * q)) : make_uint4(0, 0, 0, 0);
            a[2 * kk][e] = v.x;
            a[2 * kk][2 + e] = v.y;
            a[2 * kk + 1][e] = v.z;
            a[2 * kk + 1][2 + e] = v.w;
        }
}
__device__ __forceinline__ void tile_logits(float (&L)[RP / 8][4], const uint32_t (&a)[kD / 16][4], uint32_t zb)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < RP / 8; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) L[j][e] = 0.f;
#pragma unroll
    for (int ks = 0; ks < kD / 16; ++ks)
#pragma unroll
        for (int jp = 0; jp < RP / 16; ++jp) {
            const uint32_t off = zb + (jp * 16 + (lane & 7) + (lane >> 4) * 8) * kZPitch + (ks * 16 + ((lane >> 3) & 1) * 8) * 2;
            uint32_t bl[4], bh[4];
            logits::ldsm4(bl, off + RP * kZPitch);
            logits::ldsm4(bh, off);
            logits::mma_bf16(L[2 * jp], a[ks], bl[0], bl[1]);
            logits::mma_bf16(L[2 * jp + 1], a[ks], bl[2], bl[3]);
            logits::mma_bf16(L[2 * jp], a[ks], bh[0], bh[1]);
            logits::mma_bf16(L[2 * jp + 1], a[ks], bh[2], bh[3]);
        }
}

// The block's kernel rows around the reference potentials: to global memory, and the first ns to shared memory too (rows up to
// the next full step are zero there; the last block of the problem clears the global rows up to the next 128).
// REF: reference potentials other than one constant.  Out of line: its registers are not the iteration loop's.
template <bool REF>
__device__ __noinline__ void build16(const StreamArgs *ap, int p, int c)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const StreamArgs &a = *ap;
    const Mem m = carve16(smem, a.srows);
    const Part P = locate16(a, p, c);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
    uint32_t tok[kD / 16][4];
    fetch_tokens(tok, P, 0);
    stage_pivots(a, m, P);
    const uint32_t zb = smem_addr(m.z);
    const int direct = min(P.ns, (int)(m.z - m.K) / 128);       // rows in front of the pivots
    for (int rt = 0; rt < P.nrows; rt += 128) {
        float L[RP / 8][4];
        tile_logits(L, tok, zb);
        if (rt + 128 < P.nrows) fetch_tokens(tok, P, rt + 128);
        if (REF) {
#pragma unroll
            for (int j = 0; j < RP / 8; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) L[j][e] += (float)m.s.gref[pivot_of(j, q, e & 1)];
        }
        if (a.r < RP) {
#pragma unroll
            for (int j = 0; j < RP / 8; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (pivot_of(j, q, e & 1) >= a.r) L[j][e] = neg_inf();
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = rt + warp * 16 + g + 8 * h;
            float mx = fmaxf(L[0][2 * h], L[0][2 * h + 1]);
#pragma unroll
            for (int j = 1; j < RP / 8; ++j) mx = fmaxf(mx, fmaxf(L[j][2 * h], L[j][2 * h + 1]));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2)) - kKernelTop;
            uint32_t o[RP / 8], l[RP / 8];
#pragma unroll
            for (int j = 0; j < RP / 8; ++j) {
                const float x = ex2(L[j][2 * h] - mx), y = ex2(L[j][2 * h + 1] - mx);
                o[j] = pack2(x, y);
                l[j] = pack2(x - __uint_as_float(o[j] << 16), y - __uint_as_float(o[j] & 0xffff0000u));
            }
            if (i >= P.nrows) continue;
            // odd rows store their second half first: eight lanes then cover all banks
            const bool odd = g & 1;
            const uint4 o0 = odd ? make_uint4(o[4], o[5], o[6], o[7]) : make_uint4(o[0], o[1], o[2], o[3]);
            const uint4 o1 = odd ? make_uint4(o[0], o[1], o[2], o[3]) : make_uint4(o[4], o[5], o[6], o[7]);
            const int at = i * 128 + 16 * q + (odd ? 64 : 0), flip = odd ? -64 : 64;
            *reinterpret_cast<uint4 *>(P.g + at) = o0;
            *reinterpret_cast<uint4 *>(P.g + at + flip) = o1;
            if (i < direct) {
                *reinterpret_cast<uint4 *>(m.K + at) = o0;
                *reinterpret_cast<uint4 *>(m.K + at + flip) = o1;
            }
            if (P.low != nullptr) {                                 // read once, by the apply kernel: not to be kept in the L2
                __stcs(reinterpret_cast<uint4 *>(P.low + at), odd ? make_uint4(l[4], l[5], l[6], l[7]) : make_uint4(l[0], l[1], l[2], l[3]));
                __stcs(reinterpret_cast<uint4 *>(P.low + at + flip), odd ? make_uint4(l[0], l[1], l[2], l[3]) : make_uint4(l[4], l[5], l[6], l[7]));
            }
        }
    }
    __syncthreads();                                            // the pivots are done with
    for (int idx = direct * 8 + threadIdx.x; idx < P.steps * kRowsStep * 8; idx += kThreads)
        *reinterpret_cast<uint4 *>(m.K + idx * 16) = idx < P.ns * 8 ? __ldcg(reinterpret_cast<const uint4 *>(P.g + idx * 16)) : make_uint4(0, 0, 0, 0);
    if (c == a.C - 1) {
        const int end = min((P.nv + 127) & ~127, a.npad) - P.nv;
        uint8_t *o = a.kt + ((size_t)(P.side * a.B * a.H + P.slice) * a.npad + P.nv) * 128;
        for (int idx = threadIdx.x; idx < end * 8; idx += kThreads) *reinterpret_cast<uint4 *>(o + (size_t)idx * 16) = make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
}

// A lane's sixteen columns of a row: the 16-byte chunks cl and 4 + cl.  Lanes of odd rows read chunk 4 + cl first: the eight
// lanes of a 128-byte phase, two rows, then cover all banks without a permuted layout, and the first halving of the
// column sums is an exchange without selects.
struct LaneMap {
    uint32_t k, w, red, own;             // the second chunk of a row is at k ^ 64, its weights at w ^ 128
    int i0, at;
};

__device__ __forceinline__ LaneMap make_map16(const Mem &m)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 2;
    LaneMap L;
    const int chunk = (sub & 1) * 4 + (lane & 3);
    L.i0 = warp * 8 + sub;
    L.at = L.i0 * 128 + chunk * 16;
    L.k = smem_addr(m.K) + L.at;
    L.w = smem_addr(m.s.w) + chunk * 32;
    // after the halvings: two columns of chunk (odd, cl)
    const int col = chunk * 8 + ((lane & 8) ? 4 : 0) + ((lane & 16) ? 2 : 0);
    L.red = smem_addr(m.s.work) + (warp * RP + col) * 4;
    L.own = smem_addr(m.s.work) + threadIdx.x * 4;
    return L;
}

__device__ __forceinline__ void load_weights16(const LaneMap &L, u64 (&w)[8])
{
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        lds2(w[4 * v], w[4 * v + 1], L.w ^ (v * 128));
        lds2(w[4 * v + 2], w[4 * v + 3], (L.w ^ (v * 128)) + 16);
    }
}

// pairs of bf16 as packed float pairs
__device__ __forceinline__ u64 widen(uint32_t x) { return pack_f2(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u)); }

__device__ __forceinline__ void row16(const uint4 &a, const uint4 &b, const u64 (&w)[8], u64 (&acc)[8])
{
    const u64 k[8] = {widen(a.x), widen(a.y), widen(a.z), widen(a.w), widen(b.x), widen(b.y), widen(b.z), widen(b.w)};
    u64 s0 = 0, s1 = 0;
#pragma unroll
    for (int j = 0; j < 8; j += 2) { s0 = fma_f2(k[j], w[j], s0); s1 = fma_f2(k[j + 1], w[j + 1], s1); }
    float x, y, u, v;
    unpack_f2(s0, x, y);
    unpack_f2(s1, u, v);
    float s = (x + y) + (u + v);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    const float inv = rcp(fmaxf(s, 1e-37f));
    const u64 ii = pack_f2(inv, inv);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = fma_f2(k[j], ii, acc[j]);
}

__device__ __forceinline__ uint4 lds4(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ uint4 ldg_or_zero(bool in, const uint8_t *p)
{
    return in ? __ldcg(reinterpret_cast<const uint4 *>(p)) : make_uint4(0, 0, 0, 0);
}

// Column sums of the block's rows.  Rows that are not in shared memory come from L2, kAhead steps requested together, with
// steps from shared memory between the request and the use.  Rows kept in registers, or the next request made before the
// last is used, take registers that the loop has not got: 8.2 us a pass at n = 16384, H = 16 against 9.1 and 10.0.
__device__ __forceinline__ void pass16(const LaneMap &L, const Part &P, const u64 (&w)[8], u64 (&acc)[8])
{
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0;
    constexpr int kAhead = 2;
    uint32_t k = L.k;
    const uint32_t end = k + P.steps * (kRowsStep * 128);
    int left = P.nrows - P.ns;
    if (left > 0) {
        const uint8_t *g = P.g + (size_t)(P.nrows - left) * 128 + L.at;
        const int flip = 64 - 2 * (L.at & 64);
        const uint32_t between = (P.steps / ((left + kAhead * kRowsStep - 1) / (kAhead * kRowsStep))) * (kRowsStep * 128);
#pragma unroll 1
        for (; left > 0; left -= kAhead * kRowsStep, g += kAhead * kRowsStep * 128) {
            uint4 ra[kAhead], rb[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const bool in = u * kRowsStep + L.i0 < left;
                ra[u] = ldg_or_zero(in, g + u * (kRowsStep * 128));
                rb[u] = ldg_or_zero(in, g + u * (kRowsStep * 128) + flip);
            }
#pragma unroll 1
            for (const uint32_t stop = k + between; k < stop; k += kRowsStep * 128) row16(lds4(k), lds4(k ^ 64), w, acc);
#pragma unroll
            for (int u = 0; u < kAhead; ++u) row16(ra[u], rb[u], w, acc);
        }
    }
#pragma unroll 1
    for (; k + kRowsStep * 128 < end; k += 2 * kRowsStep * 128) {
        const uint4 a0 = lds4(k), b0 = lds4(k ^ 64), a1 = lds4(k + kRowsStep * 128), b1 = lds4((k ^ 64) + kRowsStep * 128);
        row16(a0, b0, w, acc);
        row16(a1, b1, w, acc);
    }
    if (k < end) row16(lds4(k), lds4(k ^ 64), w, acc);
}

// One iteration, as in lot_sweep_core.cuh: the weights in shared memory and those before them.
template <bool GROUP>
__device__ __forceinline__ bool iterate16(const StreamArgs &a, const Mem &m, const Part &P, const LaneMap &L, u64 (&w)[8], int group, int c,
                                          unsigned &seq)
{
    u64 acc[8];
    pass16(L, P, w, acc);
    float v[16];
#pragma unroll
    for (int j = 0; j < 8; ++j) unpack_f2(acc[j], v[2 * j], v[2 * j + 1]);
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[8 + i], 4);       // even rows keep chunk cl, odd ones 4 + cl
#pragma unroll
    for (int h = 4, bit = 8; h >= 2; h >>= 1, bit <<= 1) {
        const bool up = (lane & bit) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float give = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, bit);
        }
    }
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(L.red), "f"(v[0]), "f"(v[1]) : "memory");
    __syncthreads();
    float tot = 0.f;
    if (threadIdx.x < RP) {
        float o[kThreads / 32];
#pragma unroll
        for (int i = 0; i < kThreads / 32; ++i) o[i] = lds(L.own + i * (RP * 4));
#pragma unroll
        for (int h = kThreads / 64; h > 0; h >>= 1)
#pragma unroll
            for (int i = 0; i < h; ++i) o[i] += o[i + h];
        tot = o[0];
    }
    if (GROUP) tot = group_columns<RP, kThreads, false>(a, m.s, tot, group, c, seq);
    if ((int)threadIdx.x < a.r) {
        const float wnew = m.s.tgt[threadIdx.x] * rcp(tot);
        if (out_of_range(wnew)) m.s.flag[1] = 1;
        m.before[threadIdx.x] = m.s.w[threadIdx.x];
        m.s.w[threadIdx.x] = wnew;
    }
    __syncthreads();
    load_weights16(L, w);
    return m.s.flag[1] != 0;
}

// Whether the weights spread over more than the 60 binades the apply kernels take (the same answer in every thread).
__device__ __forceinline__ bool too_wide(const Mem &m, int r)
{
    float lo = 3e38f, hi = 0.f;
    for (int t = threadIdx.x & 31; t < r; t += 32) {
        const float w = m.s.w[t];
        lo = fminf(lo, w);
        hi = fmaxf(hi, w);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
    }
    return hi * 8.6736174e-19f > lo;
}

// log2 of the column sums of the row-stochastic plan for the potentials in gref, in the log domain: logits once for the
// column maxima and once more for the sums relative to them; nothing is stored.
template <bool GROUP>
__device__ __forceinline__ float log_columns16(const StreamArgs &a, const Mem &m, const Part &P, int group, int c, unsigned &seq)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
    float *red = reinterpret_cast<float *>(m.s.work);
    float kap = 0.f, out = 0.f;
#pragma unroll 1
    for (int round = 0; round < 2; ++round) {
        float col[RP / 8][2];
#pragma unroll
        for (int j = 0; j < RP / 8; ++j) { col[j][0] = round == 0 ? neg_inf() : 0.f; col[j][1] = col[j][0]; }
        stage_pivots(a, m, P);
        for (int rt = 0; rt < P.nrows; rt += 128) {
            uint32_t tok[kD / 16][4];
            fetch_tokens(tok, P, rt);
            float L[RP / 8][4];
            tile_logits(L, tok, smem_addr(m.z));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool ok = rt + warp * 16 + g + 8 * h < P.nrows;
                float mx = neg_inf(), s = 0.f;
#pragma unroll
                for (int j = 0; j < RP / 8; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int t = pivot_of(j, q, e);
                        L[j][2 * h + e] = t < a.r ? L[j][2 * h + e] + (float)m.s.gref[t] : neg_inf();
                        mx = fmaxf(mx, L[j][2 * h + e]);
                    }
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
#pragma unroll
                for (int j = 0; j < RP / 8; ++j) s += ex2(L[j][2 * h] - mx) + ex2(L[j][2 * h + 1] - mx);
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                const float M = mx + lg2(s);
                if (ok) {
#pragma unroll
                    for (int j = 0; j < RP / 8; ++j)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float x = L[j][2 * h + e] - M;
                            if (round == 0) col[j][e] = fmaxf(col[j][e], x);
                            else if (m.before[pivot_of(j, q, e)] > neg_inf()) col[j][e] += ex2(x - m.before[pivot_of(j, q, e)]);
                        }
                }
            }
        }
#pragma unroll
        for (int j = 0; j < RP / 8; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float v = col[j][e];
#pragma unroll
                for (int off = 4; off < 32; off <<= 1) {
                    const float o = __shfl_xor_sync(0xffffffffu, v, off);
                    v = round == 0 ? fmaxf(v, o) : v + o;
                }
                if (g == 0) red[warp * RP + pivot_of(j, q, e)] = v;
            }
        __syncthreads();
        float tot = round == 0 ? neg_inf() : 0.f;
        if (threadIdx.x < RP)
            for (int w = 0; w < kThreads / 32; ++w) tot = round == 0 ? fmaxf(tot, red[w * RP + threadIdx.x]) : tot + red[w * RP + threadIdx.x];
        if (GROUP) tot = round == 0 ? group_columns<RP, kThreads, true>(a, m.s, tot, group, c, seq) : group_columns<RP, kThreads, false>(a, m.s, tot, group, c, seq);
        __syncthreads();
        if (round == 0) {
            kap = tot;
            if (threadIdx.x < RP) m.before[threadIdx.x] = kap;      // the maxima
        } else {
            out = kap + lg2(tot);
        }
        __syncthreads();
    }
    return out;
}

// The iterations of a problem on the kernel as built.  flag[2] = 1 where recover16 has to go on from iteration flag[3].
// Returns the sequence number.
template <bool GROUP>
__device__ __noinline__ unsigned solve16(const StreamArgs *ap, int p, int group, int c, unsigned seq)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const StreamArgs &a = *ap;
    const Mem m = carve16(smem, a.srows);
    const Part P = locate16(a, p, c);
    bool bad = false;
    int it = 0;
    const LaneMap L = make_map16(m);
    u64 w[8];
    load_weights16(L, w);
    for (; it < a.T; ++it) {
        bad = iterate16<GROUP>(a, m, P, L, w, group, c, seq);
        if (bad) break;
    }
    bad = bad || too_wide(m, a.r);
    if (threadIdx.x == 0) { m.s.flag[2] = bad; m.s.flag[3] = it; }
    __syncthreads();
    return seq;
}

// The rest of a problem's iterations behind an update that left the kernel's range, as recover() of the sweep kernels; and the
// rebuilding around final potentials that spread too far for the apply kernels.
template <bool GROUP>
__device__ __noinline__ unsigned recover16(const StreamArgs *ap, int p, int group, int c, unsigned seq)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const StreamArgs &a = *ap;
    const Mem m = carve16(smem, a.srows);
    const Part P = locate16(a, p, c);
    const int tid = threadIdx.x, r = a.r;
    const float tgt = m.s.tgt[tid < RP ? tid : 0];
    int it = m.s.flag[3];
    while (true) {
        double gn = 0.0;
        const float wold = m.before[tid < RP ? tid : 0], wnew = m.s.w[tid < RP ? tid : 0];
        if (__syncthreads_or(tid < r && it < a.T && sum_lost(tgt, wnew))) {
            if (tid < r) {
                gn = m.s.gref[tid] + log2((double)wold);
                m.s.gref[tid] = gn;
            }
            __syncthreads();
            const float lam = log_columns16<GROUP>(a, m, P, group, c, seq);
            if (tid < r) gn += log2((double)tgt) - (double)lam;
        } else if (tid < r) {
            gn = m.s.gref[tid] + log2((double)wnew);
        }
        __syncthreads();
        if (tid < RP) {
            if (tid < r && !isfinite(gn)) atomicOr(a.status, 1 /* LOT_DEV_NONFINITE */);
            m.s.gref[tid] = gn - (double)kStartLog2;
            m.s.w[tid] = tid < r ? kStart : 0.f;
        }
        if (tid == 0) m.s.flag[1] = 0;
        __syncthreads();
        build16<true>(ap, p, c);
        bool bad = false;
        const LaneMap L = make_map16(m);
        u64 w[8];
        load_weights16(L, w);
        if (it >= a.T) break;                                // rebuilt around the final potentials: equal weights
        for (++it; it < a.T && !bad; ++it) bad = iterate16<GROUP>(a, m, P, L, w, group, c, seq);
        if (bad) --it;                                       // the iteration whose update has to be redone
        else if (!too_wide(m, r)) break;
        __syncthreads();
    }
    return seq;
}

template <bool GROUP>
__global__ void __launch_bounds__(kThreads, 2)
stream_kernel(const __grid_constant__ StreamArgs a)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, group = GROUP ? blockIdx.x / a.C : blockIdx.x, c = GROUP ? blockIdx.x % a.C : 0;
    unsigned seq = 0;
    const Mem m = carve16(smem, a.srows);
    if (tid < 4) m.s.flag[tid] = 0;
    if (GROUP) open_exchange<RP>(a, m.s);

    for (int p = group; p < 2 * a.B * a.H; p += a.groups) {
        __syncthreads();                                            // the previous problem is done with shared memory
        if (tid < RP) {
            const Part F = locate16(a, p, c);
            m.s.gref[tid] = -(double)kStartLog2;
            m.s.w[tid] = tid < a.r ? kStart : 0.f;
            m.before[tid] = 0.f;
            m.s.tgt[tid] = tid < a.r ? __ldg(a.beta + F.h * a.r + tid) * (float)F.nv : 0.f;
        }
        if (tid == 0) m.s.flag[2] = 0;
        if (locate16(a, p, c).nv > 0) {
            build16<false>(&a, p, c);
            seq = solve16<GROUP>(&a, p, group, c, seq);
            if (m.s.flag[2]) seq = recover16<GROUP>(&a, p, group, c, seq);
        } else {
            if (tid == 0 && c == 0) atomicOr(a.status, 2 /* LOT_DEV_EMPTY */);
            __syncthreads();
        }
        if (p + a.groups >= 2 * a.B * a.H) chain_next();
        if (c == 0 && tid < RP) {
            const Part F = locate16(a, p, c);
            const size_t sp = (size_t)F.side * a.B * a.H + F.slice;
            a.G[sp * RP + tid] = tid < a.r ? lg2(m.s.w[tid]) : 0.f;
            if (tid == 0) a.decision[sp] = 1;
            if (tid < a.r && a.g_out[F.side] != nullptr)
                a.g_out[F.side][(size_t)F.slice * a.r + tid] = (float)((m.s.gref[tid] + log2((double)m.s.w[tid])) * a.eps_ln2);
        }
    }
    if (GROUP) close_exchange(a);
}

} // namespace stream

StreamPlan stream_plan(int BH, int n)
{
    using namespace stream;
    const int NP = 2 * BH, sms = device_sm_count(), slots = 2 * sms;
    // asked for by the workspace query and by every call: the last answers are kept
    struct Memo { int BH, n, sms; StreamPlan plan; };
    static thread_local Memo memos[4] = {};
    static thread_local unsigned next = 0;
    for (const Memo &m : memos)
        if (m.BH == BH && m.n == n && m.sms == sms) return m.plan;
    StreamPlan L;
    const long long npad = ((long long)n + 127) / 128 * 128;
    // problems in flight: all of them, or as many as keep what is iterated on in the L2
    long long fly = 80000000ll / (npad * 128);
    if (fly < 2) fly = 2;
    if (fly > NP) fly = NP;
    const int rounds = (int)((NP + fly - 1) / fly), most = (n + 2 * kRowsStep - 1) / (2 * kRowsStep);
    fly = (NP + rounds - 1) / rounds;
    // Blocks a problem and blocks a cluster: the least modelled time of a call of ten iterations, us: steps of 64 rows (more where two blocks share
    // an SM), rows behind shared memory, the exchange (group_columns: one cluster; else words through L2, sixteen waited for at once,
    // behind the sums of each cluster of more than one block), and the building; at least two steps a block.  Fitted to 42 sizes
    // from one slice of 1000 tokens to three of 100000 and 400 of 600 in up to 60 forced splits: 0.7 % above the best of them on average, 7
    // at most.  Single blocks exchanging through L2 beat clusters of two where a problem has few (12 slices of 9000 tokens 87 / 94), clusters
    // of eight beat clusters of two and four where those would leave more than 16 words (one of 16384 91 / 108, of 65536 122 / 134).
    L.C = 1; L.K = 1;
    double best = 1e30;
    auto consider = [&](int C, int K, int blocks) {
        if (C > 1 && (C > most || blocks / C < 1)) return;
        const int groups = C == 1 ? (NP < blocks ? NP : blocks) : (blocks / C < NP ? blocks / C : NP), words = C / K;
        if (groups > fly) return;
        const int rows = (n + C - 1) / C, steps = (rows + kRowsStep - 1) / kRowsStep, turns = (NP + groups - 1) / groups;
        const int rest = rows > kRowsCap ? (rows - kRowsCap + kRowsStep - 1) / kRowsStep : 0;
        const bool two = groups * C > sms;
        const double lat = C == 1 ? 0.465 : C == K ? 1.1 + 0.018 * (K - 2) : 1.8 + 0.0127 * (words - 2) + 0.477 * ((words - 1) / kWords) + (K > 1 ? 1.05 : 0.0);
        const double it = lat + steps * (two ? 0.278 : 0.2) + rest * (two ? 0.089 : 0.0445);
        const double t = turns * (10.5 * it + steps * 0.68 + 4.1);
        if (t < best) { best = t; L.C = C; L.K = K; L.groups = groups; }
    };
    consider(1, 1, slots);
    for (int K = 1; K <= kPeers; ++K) {
        const int blocks = K == 1 ? slots : cluster_blocks(K, 2);
        if (K > 1) consider(K, K, blocks);
        if ((K & (K - 1)) == 0)
            for (int M = 2; M <= kMostWords && M * K <= blocks; ++M) consider(M * K, K, blocks);
    }
    if (L.C == 1) L.groups = NP;
    const int rows = (n + L.C - 1) / L.C, up = (rows + kRowsStep - 1) / kRowsStep * kRowsStep;
    L.srows = up < kRowsCap ? up : kRowsCap;
    L.npad = (int)npad;
    size_t o = 256;
    auto take = [&](size_t bytes) { const size_t at = o; o += (bytes + 255) & ~(size_t)255; return at; };
    L.xbuf = take(exchange_bytes(RP, L.C, L.K, L.groups));
    L.head_end = o;
    L.G = take((size_t)NP * RP * 4);
    L.decision = take((size_t)NP * 4);
    L.kt = take((size_t)NP * npad * 128);
    L.wpart = take(stored_apply_wpart_bytes(BH, 1, n));
    L.total = o;
    memos[next++ % 4] = Memo{BH, n, sms, L};
    return L;
}

cudaError_t stream_attention(const void *q, const void *k, const void *v, const float *z, const float *beta, const int32_t *key_len, int B,
                             int H, int n, int r, float eps, int iters, void *out, float *g1_out, float *g2_out, void *ws, cudaStream_t st)
{
    using namespace stream;
    const StreamPlan L = stream_plan(B * H, n);
    char *w = static_cast<char *>(ws);
    cudaError_t e = cudaMemsetAsync(ws, 0, L.head_end, st);
    if (e != cudaSuccess) return e;
    StreamArgs a{};
    a.x[0] = static_cast<const __nv_bfloat16 *>(q); a.x[1] = static_cast<const __nv_bfloat16 *>(k);
    a.z = z; a.beta = beta; a.key_len = key_len;
    a.kt = reinterpret_cast<uint8_t *>(w + L.kt);
    // Where the streamed path would apply from the logits, the key side is applied from twice bf16's precision.  The low
    // half waits in the output's own memory: the last kernel, which writes the output, starts behind its only reader.
    const bool low_half = !fused_ext_apply(B, H, n, r, iters);
    a.low = low_half ? static_cast<uint8_t *>(out) : nullptr;
    a.G = reinterpret_cast<float *>(w + L.G); a.decision = reinterpret_cast<int *>(w + L.decision);
    a.g_out[0] = g1_out; a.g_out[1] = g2_out;
    a.xbuf = reinterpret_cast<u64 *>(w + L.xbuf);
    a.status = reinterpret_cast<int *>(ws);
    a.B = B; a.H = H; a.n = n; a.npad = L.npad; a.r = r; a.T = iters; a.C = L.C; a.K = L.K; a.groups = L.groups; a.srows = L.srows;
    a.scale = 1.4426950408889634 / (double)eps;
    a.eps_ln2 = (double)eps * 0.6931471805599453;
    const size_t smem = (size_t)area_bytes(L.srows) + kFixed;
    const dim3 grid((unsigned)(L.C * L.groups));
    auto kern = L.C > 1 ? stream_kernel<true> : stream_kernel<false>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 113 * 1024);
    if (e != cudaSuccess) return e;
    e = L.C == L.K ? cluster_launch(kern, grid, kThreads, smem, L.K, st, a) : group_launch(kern, grid, kThreads, smem, L.K, st, a);
    if (e != cudaSuccess) return e;
    return stored_apply(a.kt, L.npad, a.G, beta, key_len, a.decision, v, out, low_half, reinterpret_cast<float *>(w + L.wpart), a.status, B, H, n, r, st);
}

} // namespace lot
