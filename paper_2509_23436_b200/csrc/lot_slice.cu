// Slice path of the LOT attention forward (Eq. (1)-(4)), one launch: a pair of thread blocks (a cluster) per (batch, head)
// slice, for sequences short enough that one side's float32 Gibbs kernel fits a block's shared memory (bf16 tensors,
// d = 64, r <= 64, n <= 512, 16 ceil(n/16) x rpad <= 16384).  One block solves the key side and the other, at the same
// time, the query side; only W' = Diag(1/beta) Gamma2 V crosses, read out of the key block's shared memory.  Nothing but
// the inputs and the output touches global memory.
//   both:     logits X Z^T * log2(e)/eps by warp-level products (Z as bf16 hi + lo), stabilised kernel to shared memory,
//             iterations and closing update as in lot_sweep.cu (lot_sweep_core.cuh)
//             with the plan rows left in the kernel's place as bf16 hi + lo
//   keys:     W = Gamma2^T V on the tensor cores
//   queries:  out = R1 W' on the tensor cores
// What bounds it: the iterations, i.e. their latency for few or short slices (about 0.7 us each) and issue slots when
// three blocks share an SM.  With the sides one after the other in one block of 512 threads the DeiT shape (B32 H3 n197
// r16 T10) took 26.7 us and the BERT shape (B16 H12 n512 r32 T20) 137 us.
#include "lot_sweep_core.cuh"

#include <mutex>

namespace lot {
namespace slice {

using namespace sweep;

constexpr int kThreads = 256, kD = 64;
constexpr int kKT = 32;                // keys per step of the W product
constexpr int kPitch = 144;            // bytes per 64-element bf16 row in shared memory (128 + 16: conflict-free ldmatrix)

struct SliceParams {
    SweepArgs s;
    const __nv_bfloat16 *v;
    __nv_bfloat16 *out;
};

template <int RP> struct Mem {
    static constexpr int z = 2 * RP * kPitch;                                       // staged pivots (hi, lo); later W' (hi, lo)
    static constexpr int v = 2 * kKT * kPitch;                                      // two steps of values
    static constexpr int red = 8 * RP * 4 * 2;
    static constexpr int slow = (int)work_bytes<__nv_bfloat16>(RP, kThreads);
    static constexpr int mx(int a, int b) { return a > b ? a : b; }
    static constexpr int work = mx(mx(z, v), mx(red, slow));
    static constexpr int ref = kTileRows(kThreads) * (RP / rebuild_cols(RP)) * 4;
    static constexpr int fixed = work + ref + RP * 16 + 64;
};

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&t);
}
// (hi, lo) bf16 pairs of two floats: x = hi + lo to about 2^-17
__device__ __forceinline__ void split2(float x0, float x1, uint32_t &hi, uint32_t &lo)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = pack2(x0 - __low2float(h), x1 - __high2float(h));
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void cluster_arrive_wait()
{
    asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
}

// The side's stabilised kernel (starting potentials zero) into S.K; rows beyond nv, up to the next full step, are zero.
template <int RP, int CPL>
__device__ __forceinline__ void first_kernel(const SweepArgs &a, int p, const Shared &S, Share &R, Problem &Q)
{
    typedef Lay<RP, CPL> Y;
    constexpr int STEP = (kThreads / 32) * Y::RPW;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;
    // every load that depends on nothing goes out before the first one is waited for: the slice's first token tile, the
    // pivots, their masses, the key length
    const int r = a.r, n = a.n[0], slice = p >> 1, h = slice % a.H;
    const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(a.x[(p & 1) ^ 1]) + (size_t)slice * n * kD;
    const float *z = a.z + (size_t)h * r * kD;
    const float scale = (float)a.scale;
    uint32_t xa[kD / 16][4];
    auto fetch = [&](int rt) {
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int i = rt + warp * 16 + g + (e & 1) * 8;
                xa[ks][e] = i < n ? __ldg(reinterpret_cast<const unsigned *>(x + (size_t)i * kD + ks * 16 + (e >> 1) * 8 + 2 * q)) : 0u;
            }
    };
    fetch(0);
    constexpr int NZ = RP * (kD / 2) / kThreads;
    float2 zz[NZ];
#pragma unroll
    for (int u = 0; u < NZ; ++u) {
        const int idx = tid + u * kThreads, t = idx / (kD / 2);
        zz[u] = t < r ? __ldg(reinterpret_cast<const float2 *>(z + (size_t)t * kD + (idx % (kD / 2)) * 2)) : make_float2(0.f, 0.f);
    }
    const float bt = tid < r ? __ldg(a.beta + h * r + tid) : 0.f;
    Q = locate<RP, CPL, kThreads>(a, p, 0, R);
    const int rows = R.steps * STEP;
    if (tid < RP) {
        S.gref[tid] = -(double)kStartLog2;
        S.w[tid] = tid < r ? kStart : 0.f;
        S.tgt[tid] = bt * (float)Q.nv;
    }
    // pivots of this head in base-2 logit units, bf16 hi + lo
#pragma unroll
    for (int u = 0; u < NZ; ++u) {
        const int idx = tid + u * kThreads, t = idx / (kD / 2), c2 = (idx % (kD / 2)) * 2;
        uint32_t hi, lo;
        split2(zz[u].x * scale, zz[u].y * scale, hi, lo);
        *reinterpret_cast<uint32_t *>(S.work + t * kPitch + c2 * 2) = hi;
        *reinterpret_cast<uint32_t *>(S.work + (RP + t) * kPitch + c2 * 2) = lo;
    }
    __syncthreads();
    const uint32_t zb = smem_addr(S.work);
    for (int rt = 0; rt < rows; rt += 128) {
        float L[RP / 8][4];
#pragma unroll
        for (int j = 0; j < RP / 8; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) L[j][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks)
#pragma unroll
            for (int jp = 0; jp < RP / 16; ++jp) {
                const uint32_t off = zb + (jp * 16 + (lane & 7) + (lane >> 4) * 8) * kPitch + (ks * 16 + ((lane >> 3) & 1) * 8) * 2;
                uint32_t bl[4], bh[4];
                logits::ldsm4(bl, off + RP * kPitch);
                logits::ldsm4(bh, off);
                logits::mma_bf16(L[2 * jp], xa[ks], bl[0], bl[1]);
                logits::mma_bf16(L[2 * jp + 1], xa[ks], bl[2], bl[3]);
                logits::mma_bf16(L[2 * jp], xa[ks], bh[0], bh[1]);
                logits::mma_bf16(L[2 * jp + 1], xa[ks], bh[2], bh[3]);
            }
        if (rt + 128 < rows) fetch(rt + 128);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = rt + warp * 16 + g + 8 * h;
            float m = neg_inf();
#pragma unroll
            for (int j = 0; j < RP / 8; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (8 * j + 2 * q + e >= r) L[j][2 * h + e] = neg_inf();
                    m = fmaxf(m, L[j][2 * h + e]);
                }
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2)) - kKernelTop;
            if (i < rows) {
#pragma unroll
                for (int j = 0; j < RP / 8; ++j) {
                    const int c0 = 8 * j + 2 * q;
                    float2 v = make_float2(0.f, 0.f);
                    if (i < R.nrows) v = make_float2(ex2(L[j][2 * h] - m), ex2(L[j][2 * h + 1] - m));
                    *reinterpret_cast<float2 *>(S.K + (size_t)i * RP + Y::swz(i, c0 >> 2) * 4 + (c0 & 3)) = v;
                }
            }
        }
    }
    __syncthreads();
}

// Closing update in place: kernel rows become plan rows R_it = K_it w_t / s_i, as bf16 hi + lo: a 16-byte chunk of four
// pivots then holds their four hi parts and their four lo parts, which the products below take as eight "pivots".
template <int RP, int CPL>
__device__ __forceinline__ void close_rows(const Shared &S, const Share &R)
{
    typedef Lay<RP, CPL> Y;
    constexpr int STEP = (kThreads / 32) * Y::RPW;
    const Lane<RP, CPL> L = make_lane<RP, CPL, kThreads>(S, 0);
    u64 w[CPL / 2];
    load_weights<RP, CPL>(L, w);
    for (int st = 0; st < R.steps; ++st) {
        Row<CPL> k;
        u64 none[CPL / 2];
#pragma unroll
        for (int v = 0; v < Y::NV; ++v) lds2(k.k[2 * v], k.k[2 * v + 1], L.k[v] + st * (STEP * RP * 4));
        const float inv = row_step<RP, CPL, false>(k, w, none, 1.f);
#pragma unroll
        for (int v = 0; v < Y::NV; ++v) {
            float2 x, y, wx, wy;
            unpack_f2(k.k[2 * v], x.x, x.y);
            unpack_f2(k.k[2 * v + 1], y.x, y.y);
            unpack_f2(w[2 * v], wx.x, wx.y);
            unpack_f2(w[2 * v + 1], wy.x, wy.y);
            uint32_t h0, l0, h1, l1;
            split2((x.x * inv) * wx.x, (x.y * inv) * wx.y, h0, l0);
            split2((y.x * inv) * wy.x, (y.y * inv) * wy.y, h1, l1);
            asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(L.k[v] + st * (STEP * RP * 4)), "r"(h0), "r"(h1), "r"(l0), "r"(l1) : "memory");
        }
    }
    __syncthreads();
}

template <int RP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, max_blocks(wide_cols(RP), kThreads))
slice_forward_kernel(const __grid_constant__ SliceParams P)
{
    constexpr int CPL = wide_cols(RP);
    typedef Lay<RP, CPL> Y;
    extern __shared__ __align__(1024) uint8_t smem[];
    const SweepArgs &a = P.s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3, mi = lane >> 3;
    const int p = blockIdx.x, n = a.n[0], r = a.r;                 // p even: keys, odd: queries of slice p / 2
    const Shared S = carve<__nv_bfloat16, RP, kThreads>(smem, a.srows, Mem<RP>::work, Mem<RP>::ref);
    Share R;
    Problem Q;
    if (tid == 0) { S.flag[0] = 0; S.flag[1] = 0; }
    first_kernel<RP, CPL>(a, p, S, R, Q);
    const float *beta = a.beta + Q.h * r;
    const size_t tok = (size_t)Q.slice * n * kD;
    if (Q.nv > 0) {
        float wold = 0.f, wnew = S.w[tid < RP ? tid : 0];
        bool bad = false;
        int it = 0;
        unsigned seq = 0;
        {
            const Lane<RP, CPL> L = make_lane<RP, CPL, kThreads>(S, 0);
            const float tgt = S.tgt[tid < RP ? tid : 0];
            u64 w[CPL / 2];
            load_weights<RP, CPL>(L, w);
            for (; it < a.iters; ++it) {
                bad = iterate<RP, CPL, kThreads, false, false>(a, S, R, L, w, tgt, 0, 0, seq, wold, wnew);
                if (bad) break;
            }
        }
        if (bad) recover<__nv_bfloat16, RP, CPL, kThreads, false, false, Mem<RP>::work, Mem<RP>::ref>(&a, p, 0, 0, it, seq, wold, wnew);
        close_rows<RP, CPL>(S, R);
    } else {
        // no keys: nothing to transport; the output is zero (flagged), the key-side potentials stay at zero
        if (tid == 0) atomicOr(a.status, 2 /* LOT_DEV_EMPTY */);
        if (tid < RP) { S.gref[tid] = 0.0; S.w[tid] = 1.f; }
        __syncthreads();
    }
    if (tid < r && a.g_out[Q.side] != nullptr)
        a.g_out[Q.side][(size_t)Q.slice * r + tid] = (float)((S.gref[tid] + log2((double)S.w[tid])) * a.eps_ln2);

    float *sWf = S.K;                                              // keys: W' as [RP][64] floats, once the kernel is used up
    if (Q.side == 1) {
        // W[t][c] = sum_j R2[j][t] v[j][c]: warps are tiles of eight pivots (16 rows: hi and lo parts) x channel groups; the
        // values come through shared memory, kKT keys at a time, two steps in flight
        constexpr int MT = RP / 8, CG = 8 / MT, NTW = 8 / CG;
        const int mt = warp % MT, cg = warp / MT;
        const __nv_bfloat16 *V = P.v + tok;
        const uint32_t vb = smem_addr(S.work), kb = smem_addr(S.K);
        float acc[NTW][4] = {};
        auto fetch = [&](int j0, int buf) {
            const int j = j0 + tid / 8;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\ncp.async.commit_group;" ::"r"(vb + (buf * kKT + tid / 8) * kPitch + (tid % 8) * 16),
                         "l"(V + (size_t)min(j, n - 1) * kD + (tid % 8) * 8), "r"(j < Q.nv ? 16 : 0) : "memory");
        };
        fetch(0, 0);
        int buf = 0;
        for (int j0 = 0; j0 < Q.nv; j0 += kKT, buf ^= 1) {
            fetch(j0 + kKT, buf ^ 1);                              // past the end: zeros
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncthreads();
#pragma unroll
            for (int s = 0; s < kKT / 16; ++s) {
                const int j = j0 + s * 16 + (lane & 7) + (mi >> 1) * 8;
                if (j0 + s * 16 >= R.steps * ((kThreads / 32) * Y::RPW)) break;
                uint32_t af[4];
                ldsm4_t(af, kb + (j * Y::CH + Y::swz(j, mt * 2 + (mi & 1))) * 16);
#pragma unroll
                for (int nt = 0; nt < NTW; nt += 2) {
                    uint32_t bv[4];
                    ldsm4_t(bv, vb + (buf * kKT + s * 16 + (lane & 7) + (mi & 1) * 8) * kPitch + (cg * NTW * 8 + nt * 8 + (mi >> 1) * 8) * 2);
                    logits::mma_bf16(acc[nt], af, bv[0], bv[1]);
                    logits::mma_bf16(acc[nt + 1], af, bv[2], bv[3]);
                }
            }
            __syncthreads();
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        const float ikv = Q.nv > 0 ? 1.f / (float)Q.nv : 0.f;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int t = mt * 8 + hh * 4 + (g & 3);
            const float f = t < r ? ikv / __ldg(beta + t) : 0.f;
#pragma unroll
            for (int nt = 0; nt < NTW; ++nt) {
                float2 v = make_float2(acc[nt][2 * hh], acc[nt][2 * hh + 1]);
                v.x += __shfl_xor_sync(0xffffffffu, v.x, 16);      // hi + lo
                v.y += __shfl_xor_sync(0xffffffffu, v.y, 16);
                if (g < 4) *reinterpret_cast<float2 *>(sWf + t * kD + cg * NTW * 8 + nt * 8 + 2 * q) = make_float2(v.x * f, v.y * f);
            }
        }
    }
    cluster_arrive_wait();                                         // W' is complete, the query block has its plan
    if (Q.side == 0) {
        // W' out of the key block's shared memory, as bf16 hi + lo planes [pivot][channel]
        uint32_t remote;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_addr(sWf)), "r"(0));
        for (int idx = tid; idx < RP * kD / 4; idx += kThreads) {
            float4 v;
            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(remote + idx * 16) : "memory");
            uint2 hi, lo;
            split2(v.x, v.y, hi.x, lo.x);
            split2(v.z, v.w, hi.y, lo.y);
            uint8_t *o = S.work + (idx / (kD / 4)) * kPitch + (idx % (kD / 4)) * 8;
            *reinterpret_cast<uint2 *>(o) = hi;
            *reinterpret_cast<uint2 *>(o + RP * kPitch) = lo;
        }
    }
    cluster_arrive_wait();                                         // the key block may go, the planes are in place
    if (Q.side == 1) return;
    // out[i][c] = sum_t R1[i][t] W'[t][c]
    __nv_bfloat16 *ob = P.out + tok;
    for (int rt = warp * 16; rt < n; rt += 128) {
        float acc[kD / 8][4] = {};
        for (int k = 0; k < RP / 8; ++k) {                         // eight pivots: hi and lo parts against the same W' rows
            uint32_t af[4], bh[4], bl[4];
            const int i = rt + (lane & 7) + (mi & 1) * 8;
            logits::ldsm4(af, smem_addr(S.K) + (i * Y::CH + Y::swz(i, k * 2 + (mi >> 1))) * 16);
#pragma unroll
            for (int cp = 0; cp < kD / 16; ++cp) {
                // operand rows 0-3 and 4-7 are the same four pivots, likewise 8-11 and 12-15
                const int t = k * 8 + (lane & 3) + (mi & 1) * 4;
                const uint32_t off = smem_addr(S.work) + t * kPitch + (cp * 16 + (mi >> 1) * 8) * 2;
                ldsm4_t(bl, off + RP * kPitch);
                ldsm4_t(bh, off);
                logits::mma_bf16(acc[2 * cp], af, bl[0], bl[1]);
                logits::mma_bf16(acc[2 * cp + 1], af, bl[2], bl[3]);
                logits::mma_bf16(acc[2 * cp], af, bh[0], bh[1]);
                logits::mma_bf16(acc[2 * cp + 1], af, bh[2], bh[3]);
            }
        }
        // neighbouring lanes trade halves of neighbouring channel tiles: a quad then stores 32 consecutive bytes of a row
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int i = rt + g + 8 * hh;
#pragma unroll
            for (int j = 0; j < kD / 8; j += 2) {
                const uint32_t u0 = pack2(acc[j][2 * hh], acc[j][2 * hh + 1]), u1 = pack2(acc[j + 1][2 * hh], acc[j + 1][2 * hh + 1]);
                const uint32_t got = __shfl_xor_sync(0xffffffffu, q & 1 ? u0 : u1, 1);
                const uint2 o = q & 1 ? make_uint2(got, u1) : make_uint2(u0, got);
                if (i < n) *reinterpret_cast<uint2 *>(ob + (size_t)i * kD + 8 * (j + (q & 1)) + 4 * (q >> 1)) = o;
            }
        }
    }
}

template <int RP>
cudaError_t launch(SliceParams P, int BH, cudaStream_t st)
{
    static std::mutex mu;
    static bool attr_set[64] = {};
    auto kern = slice_forward_kernel<RP>;
    const int step = kThreads * wide_cols(RP) / RP, n = P.s.n[0];
    int rows = (n + step - 1) / step * step;
    if (rows < kD) rows = kD;                                      // room for W'
    P.s.srows = rows;
    const size_t smem = (size_t)rows * RP * 4 + Mem<RP>::fixed;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!attr_set[dev]) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 16384 * 4 + Mem<RP>::fixed);
            if (e != cudaSuccess) return e;
            attr_set[dev] = true;
        }
    }
    kern<<<2 * BH, kThreads, smem, st>>>(P);
    return cudaGetLastError();
}

} // namespace slice

bool slice_supported(int dtype, int n, int d, int r)
{
    if (dtype != 1 || d != slice::kD || r < 1 || r > 64 || n < 1 || n > 512) return false;
    const int rp = r <= 16 ? 16 : r <= 32 ? 32 : 64;
    return ((n + 15) / 16) * 16 * rp <= 16384;
}

cudaError_t slice_attention(const void *q, const void *k, const void *v, const float *z, const float *beta,
                            const int32_t *key_len, int B, int H, int n, int r, float eps, int iters, void *out,
                            float *g1_out, float *g2_out, int *status, cudaStream_t st)
{
    slice::SliceParams P{};
    P.s.x[0] = q; P.s.x[1] = k; P.s.z = z; P.s.beta = beta; P.s.key_len = key_len;
    P.s.g_out[0] = g1_out; P.s.g_out[1] = g2_out; P.s.status = status;
    P.s.B = B; P.s.H = H; P.s.d = slice::kD; P.s.r = r; P.s.n[0] = P.s.n[1] = n;
    P.s.C = 1; P.s.groups = 2 * B * H; P.s.iters = iters;
    P.s.scale = 1.4426950408889634 / (double)eps;
    P.s.eps_ln2 = (double)eps * 0.6931471805599453;
    P.v = static_cast<const __nv_bfloat16 *>(v);
    P.out = static_cast<__nv_bfloat16 *>(out);
    cudaError_t e = cudaMemsetAsync(status, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    const int BH = B * H;
    return r <= 16 ? slice::launch<16>(P, BH, st) : r <= 32 ? slice::launch<32>(P, BH, st) : slice::launch<64>(P, BH, st);
}

} // namespace lot
