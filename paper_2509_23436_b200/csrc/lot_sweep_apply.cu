// Apply stages behind the sweep kernel (Eq. (4)): W' = Diag(1/beta) Gamma2 V and out = R1 W', with the plan rows read
// off the stored Gibbs kernel: R_it = kt_it w_t inv_i.
//
// bf16 tensors: tensor cores, warp-level products.  A float32 factor is the exact sum of three bf16 terms, so with N = 3 the
// products are those of the float32 evaluation up to terms below 2^-24 (N = 2, hi + lo: 2^-17) and sums accumulate in
// float32; the plan entries never exist in memory.  float32 tensors: CUDA cores (their products would need six terms a piece on the tensor cores).
// All kernels load the next step's operands into registers while the current one multiplies; what bounds them is the
// read of the kernel (4 bytes per entry) and, at rank 256, the product rate.
#include "lot_chain.cuh"
#include "lot_internal.h"
#include "lot_logits.cuh"
#include "lot_sweep.h"

namespace lot {
namespace sweep_apply {

constexpr int kThreads = 256;

using logits::ldsm4_t;
using logits::smem_addr;
using logits::split;

__device__ __forceinline__ float4 scaled(float4 p, float4 w, float s)
{
    return make_float4(p.x * (w.x * s), p.y * (w.y * s), p.z * (w.z * s), p.w * (w.w * s));
}

// The partials of the chunks in order, eight requested together: the last block of a tile does this alone, one L2 round
// trip after the other.
__device__ __forceinline__ float4 add_partials(const float *src, size_t stride, int chunks)
{
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0; c0 < chunks; c0 += 8) {
        float4 p[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            p[u] = c0 + u < chunks ? __ldcg(reinterpret_cast<const float4 *>(src + (size_t)(c0 + u) * stride)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u) { s.x += p[u].x; s.y += p[u].y; s.z += p[u].z; s.w += p[u].w; }
    }
    return s;
}

// The tickets of the blocks that share a tile: true in the last one to arrive, which adds the partials in chunk order.
__device__ __forceinline__ bool last_of_tile(unsigned *counter, int chunks)
{
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(counter, 1u) == (unsigned)chunks - 1u;
        if (last) *counter = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last != 0;
}

// ---------------------------------------------------------------------------------------------------------------
// Key side, bf16 tensors: W[t][c] = sum_j R_jt m_j v_jc.  Block = TP pivots x D channels over one chunk of keys, 64 keys per
// step: the plan tile goes to shared memory as N bf16 planes (transposed on the way to the tensor cores), the values
// as they are.  Warps: TP / 16 pivot tiles x channel groups x (rank 16, narrow heads) halves of the keys.
// ---------------------------------------------------------------------------------------------------------------
template <int TP, int D, int N>
__global__ void __launch_bounds__(kThreads, D <= 128 ? 2 : 1)
apply_w_mma_kernel(const __grid_constant__ SweepApplyArgs a0, const __grid_constant__ SweepApplyArgs a1)
{
    const bool second = (int)blockIdx.z >= a0.B * a0.H;            // two products of the same sizes in one launch
    const SweepApplyArgs &a = second ? a1 : a0;
    constexpr int KT = 64, PP = (TP + 8) * 2, PV = (D + 8) * 2, PLANE = KT * PP;
    constexpr int PT = TP / 16, CG = 8 / PT < D / 16 ? 8 / PT : D / 16, KS = 8 / (PT * CG), NTW = D / 8 / CG;
    constexpr int NP = KT * TP / 4 / kThreads, NV = KT * D / 8 / kThreads;
    extern __shared__ __align__(128) uint8_t sm[];
    uint8_t *sP = sm, *sV = sm + N * PLANE;
    const int bh = blockIdx.z - (second ? a0.B * a0.H : 0), b = bh / a.H, h = bh % a.H, chunk = blockIdx.x, t0 = blockIdx.y * TP;
    const int n = a.nk, r = a.r, d = a.d, RP = a.RP;
    int nv = n;
    if (a.key_len != nullptr) nv = min(max(a.key_len[b], 0), n);
    const float *mass = a.mass2 ? a.mass2 + (size_t)bh * n : nullptr;
    const float *K = a.kt[1] + (size_t)bh * n * RP + t0, *inv = a.inv[1] ? a.inv[1] + (size_t)bh * n : nullptr, *w = a.w[1] ? a.w[1] + (size_t)bh * RP + t0 : nullptr;
    const __nv_bfloat16 *V = static_cast<const __nv_bfloat16 *>(a.v) + (size_t)bh * n * d;
    const int row0 = chunk * a.rows_per_chunk + a.skip, row1 = min(min(row0 + a.rows_per_chunk, n), nv);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int pt = warp % PT, cg = (warp / PT) % CG, ks = warp / (PT * CG);

    float4 kr[NP];
    float sc[NP];
    uint4 vr[NV];
    auto fetch = [&](int j0) {
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int idx = tid + u * kThreads, j = j0 + idx / (TP / 4), t = (idx % (TP / 4)) * 4;
            kr[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            sc[u] = 0.f;
            if (j < row1) {
                kr[u] = chain_ld4(K + (size_t)j * RP + t);
                sc[u] = (inv ? chain_ld(inv + j) : 1.f) * (mass ? __ldg(mass + j) : 1.f);
            }
        }
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int idx = tid + u * kThreads, j = j0 + idx / (D / 8), c = (idx % (D / 8)) * 8;
            vr[u] = j < row1 && c < d ? __ldg(reinterpret_cast<const uint4 *>(V + (size_t)j * d + c)) : make_uint4(0, 0, 0, 0);
        }
    };
    float acc[NTW][4] = {};
    chain_wait();
    float4 wt[NP];
#pragma unroll
    for (int u = 0; u < NP; ++u)
        wt[u] = w ? chain_ld4(w + ((tid + u * kThreads) % (TP / 4)) * 4) : make_float4(1.f, 1.f, 1.f, 1.f);
    if (row0 < row1) fetch(row0);
    const int mi = lane >> 3;
    for (int j0 = row0; j0 < row1; j0 += KT) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int idx = tid + u * kThreads, j = idx / (TP / 4), t = (idx % (TP / 4)) * 4;
            const float4 p = scaled(kr[u], wt[u], sc[u]);
            uint32_t x[N], y[N];
            split<N>(p.x, p.y, x);
            split<N>(p.z, p.w, y);
#pragma unroll
            for (int i = 0; i < N; ++i) *reinterpret_cast<uint2 *>(sP + i * PLANE + j * PP + t * 2) = make_uint2(x[i], y[i]);
        }
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int idx = tid + u * kThreads;
            *reinterpret_cast<uint4 *>(sV + (idx / (D / 8)) * PV + (idx % (D / 8)) * 16) = vr[u];
        }
        __syncthreads();
        if (j0 + KT < row1) fetch(j0 + KT);
#pragma unroll
        for (int s = 0; s < KT / 16 / KS; ++s) {
            const int j = (ks * (KT / 16 / KS) + s) * 16;
            uint32_t af[N][4];
#pragma unroll
            for (int i = 0; i < N; ++i)
                ldsm4_t(af[i], smem_addr(sP) + i * PLANE + (j + (lane & 7) + (mi >> 1) * 8) * PP + (pt * 16 + (mi & 1) * 8) * 2);
#pragma unroll
            for (int nt = 0; nt < NTW; nt += 2) {
                uint32_t bf[4];
                ldsm4_t(bf, smem_addr(sV) + (j + (lane & 7) + (mi & 1) * 8) * PV + (cg * NTW * 8 + nt * 8 + (mi >> 1) * 8) * 2);
#pragma unroll
                for (int i = N - 1; i >= 0; --i) {
                    logits::mma_bf16(acc[nt], af[i], bf[0], bf[1]);
                    logits::mma_bf16(acc[nt + 1], af[i], bf[2], bf[3]);
                }
            }
        }
    }
    chain_next();
    // halves of the keys, then the chunks
    const int g = lane >> 2, q = lane & 3;
    float *red = reinterpret_cast<float *>(sm);
    if (KS > 1) {
        __syncthreads();
        if (ks > 0) {
#pragma unroll
            for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) red[(((ks - 1) * PT * CG + warp % (PT * CG)) * NTW * 4 + nt * 4 + e) * 32 + lane] = acc[nt][e];
        }
        __syncthreads();
        if (ks == 0) {
            for (int k2 = 1; k2 < KS; ++k2)
#pragma unroll
                for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[nt][e] += red[(((k2 - 1) * PT * CG + warp) * NTW * 4 + nt * 4 + e) * 32 + lane];
        }
    }
    const float scale = a.mass2 ? 1.f : (nv > a.skip ? 1.f / (float)(nv - a.skip) : 0.f);
    if (ks == 0) {
        float *wp = a.wpart + ((size_t)bh * a.chunks + chunk) * r * d, *Wp = a.Wp + (size_t)bh * r * d;
#pragma unroll
        for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int t = t0 + pt * 16 + g + 8 * hh, c = cg * NTW * 8 + nt * 8 + 2 * q;
                if (t < r && c < d) {
                    const float2 v = make_float2(acc[nt][2 * hh], acc[nt][2 * hh + 1]);
                    if (a.chunks > 1 || a.Wp == nullptr) {
                        __stcg(reinterpret_cast<float2 *>(wp + (size_t)t * d + c), v);
                    } else {
                        const float f = scale / a.beta[h * r + t];
                        *reinterpret_cast<float2 *>(Wp + (size_t)t * d + c) = make_float2(v.x * f, v.y * f);
                    }
                }
            }
    }
    if (a.chunks == 1 || a.Wp == nullptr || !last_of_tile(a.counter + (size_t)bh * gridDim.y + blockIdx.y, a.chunks)) return;
    const int nt4 = min(TP, r - t0) * d / 4;
    for (int idx = tid; idx < nt4; idx += kThreads) {
        const size_t o = (size_t)t0 * d + idx * 4;
        const float *src = a.wpart + (size_t)bh * a.chunks * r * d + o;
        const float4 s = add_partials(src, (size_t)r * d, a.chunks);
        const float f = scale / a.beta[h * r + t0 + idx * 4 / d];
        *reinterpret_cast<float4 *>(a.Wp + (size_t)bh * r * d + o) = make_float4(s.x * f, s.y * f, s.z * f, s.w * f);
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Query side, bf16 tensors: out[i][c] = sum_t R_it W'[t][c].  Block = 128 queries x D channels; a warp's 16 plan rows come
// from global memory straight into operand fragments, W' in steps of TS pivots through shared memory as N planes.
// ---------------------------------------------------------------------------------------------------------------
template <int TS, int D, int N>
__global__ void __launch_bounds__(kThreads, D <= 128 ? 2 : 1)
apply_out_mma_kernel(SweepApplyArgs a)
{
    constexpr int PW = (D + 8) * 2, PLANE = TS * PW, NW = TS * D / 4 / kThreads;
    extern __shared__ __align__(128) uint8_t sW[];
    const int bh = blockIdx.y, n = a.nq, r = a.r, d = a.d, RP = a.RP;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3, mi = lane >> 3;
    const int i0 = blockIdx.x * 128 + warp * 16 + a.skip;
    const int nrow = a.out_len ? min(max(__ldg(a.out_len + bh / a.H), 0), n) : n;     // rows beyond it are zero
    const float *K = a.kt[0] + ((size_t)bh * n + i0) * RP, *w = a.w[0] ? a.w[0] + (size_t)bh * RP : nullptr;
    const float *W = a.Wp + (size_t)(a.per_head ? bh % a.H : bh) * r * d;
    chain_wait();
    float s[2];
#pragma unroll
    for (int hh = 0; hh < 2; ++hh)
        s[hh] = i0 + g + 8 * hh < nrow ? (a.inv[0] ? chain_ld(a.inv[0] + (size_t)bh * n + i0 + g + 8 * hh) : 1.f) : 0.f;
    float2 kr[TS / 16][4];
    float4 wr[NW];
    auto fetch = [&](int tb) {
#pragma unroll
        for (int k = 0; k < TS / 16; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int row = g + (e & 1) * 8, t = tb + k * 16 + (e >> 1) * 8 + 2 * q;
                kr[k][e] = i0 + row < nrow ? chain_ld2(K + (size_t)row * RP + t) : make_float2(0.f, 0.f);
            }
#pragma unroll
        for (int u = 0; u < NW; ++u) {
            const int idx = tid + u * kThreads, t = tb + idx / (D / 4), c = (idx % (D / 4)) * 4;
            wr[u] = t < r && c < d ? chain_ld4(W + (size_t)t * d + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float acc[D / 8][4] = {};
    fetch(0);
    for (int tb = 0; tb < RP && tb < r; tb += TS) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NW; ++u) {
            const int idx = tid + u * kThreads, t = idx / (D / 4), c = (idx % (D / 4)) * 4;
            uint32_t x[N], y[N];
            split<N>(wr[u].x, wr[u].y, x);
            split<N>(wr[u].z, wr[u].w, y);
#pragma unroll
            for (int i = 0; i < N; ++i) *reinterpret_cast<uint2 *>(sW + i * PLANE + t * PW + c * 2) = make_uint2(x[i], y[i]);
        }
        uint32_t af[TS / 16][N][4];
#pragma unroll
        for (int k = 0; k < TS / 16; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 ww = w ? chain_ld2(w + tb + k * 16 + (e >> 1) * 8 + 2 * q) : make_float2(1.f, 1.f);
                uint32_t o[N];
                split<N>(kr[k][e].x * (ww.x * s[e & 1]), kr[k][e].y * (ww.y * s[e & 1]), o);
#pragma unroll
                for (int i = 0; i < N; ++i) af[k][i][e] = o[i];
            }
        __syncthreads();
        if (tb + TS < r) fetch(tb + TS);
#pragma unroll
        for (int k = 0; k < TS / 16; ++k)
#pragma unroll
            for (int cp = 0; cp < D / 16; ++cp) {
                uint32_t bf[N][4];
#pragma unroll
                for (int i = 0; i < N; ++i)
                    ldsm4_t(bf[i], smem_addr(sW) + i * PLANE + (k * 16 + (lane & 7) + (mi & 1) * 8) * PW + (cp * 16 + (mi >> 1) * 8) * 2);
#pragma unroll
                for (int o = N - 1; o >= 0; --o)                      // the products of total order o, small ones first
#pragma unroll
                    for (int i = 0; i <= o; ++i) {
                        logits::mma_bf16(acc[2 * cp], af[k][i], bf[o - i][0], bf[o - i][1]);
                        logits::mma_bf16(acc[2 * cp + 1], af[k][i], bf[o - i][2], bf[o - i][3]);
                    }
            }
    }
    chain_next();
    __nv_bfloat16 *O = static_cast<__nv_bfloat16 *>(a.out) + ((size_t)bh * n + i0) * d;
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        const int row = g + 8 * hh;
        if (i0 + row >= n) continue;
#pragma unroll
        for (int j = 0; j < D / 8; ++j)
            if (8 * j < d)
                *reinterpret_cast<__nv_bfloat162 *>(O + (size_t)row * d + 8 * j + 2 * q) = __floats2bfloat162_rn(acc[j][2 * hh], acc[j][2 * hh + 1]);
    }
}

// ---------------------------------------------------------------------------------------------------------------
// float32 tensors.  Both products have a 64-channel tile and 4 x 4 results per thread; with fewer than 64 pivots (key
// side) the spare threads take other keys of the step.
// ---------------------------------------------------------------------------------------------------------------
constexpr int kCT = 64, kStep = 32;

template <int TP>
__global__ void __launch_bounds__(kThreads, 3)
apply_w_f32_kernel(SweepApplyArgs a)
{
    constexpr int PW = TP + 4, VW = kCT + 4, GT = 16 * (TP / 4), G = kThreads / GT;     // threads per key group, key groups
    constexpr int NP = kStep * TP / 4 / kThreads < 1 ? 1 : kStep * TP / 4 / kThreads, NV = kStep * kCT / 4 / kThreads;
    __shared__ __align__(16) float Ps[kStep][PW];
    __shared__ __align__(16) float Vs[kStep][VW];
    __shared__ __align__(16) float red[G > 1 ? TP * kCT : 1];
    const int bh = blockIdx.z, b = bh / a.H, h = bh % a.H, chunk = blockIdx.x;
    const int cblks = (a.d + kCT - 1) / kCT, t0 = (blockIdx.y / cblks) * TP, c0 = (blockIdx.y % cblks) * kCT;
    const int n = a.nk, r = a.r, d = a.d, RP = a.RP, tid = threadIdx.x;
    int nv = n;
    if (a.key_len != nullptr) nv = min(max(a.key_len[b], 0), n);
    const float *mass = a.mass2 ? a.mass2 + (size_t)bh * n : nullptr;
    const float *K = a.kt[1] + (size_t)bh * n * RP + t0, *inv = a.inv[1] ? a.inv[1] + (size_t)bh * n : nullptr, *w = a.w[1] ? a.w[1] + (size_t)bh * RP + t0 : nullptr;
    const float *V = static_cast<const float *>(a.v) + (size_t)bh * n * d;
    const int row0 = chunk * a.rows_per_chunk + a.skip, row1 = min(min(row0 + a.rows_per_chunk, n), nv);
    const int grp = tid / GT, ty = (tid % GT) / 16, tx = tid % 16;
    float4 kr[NP], vr[NV], wt;
    float sc[NP];
    chain_wait();
    wt = chain_ld4(w + (tid % (TP / 4)) * 4);              // kThreads is a multiple of TP / 4
    auto fetch = [&](int j0) {
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int idx = tid + u * kThreads, j = j0 + idx / (TP / 4);
            kr[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            sc[u] = 0.f;
            if (idx < kStep * TP / 4 && j < row1) {
                kr[u] = chain_ld4(K + (size_t)j * RP + (idx % (TP / 4)) * 4);
                sc[u] = (inv ? chain_ld(inv + j) : 1.f) * (mass ? __ldg(mass + j) : 1.f);
            }
        }
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int idx = tid + u * kThreads, j = j0 + idx / 16, c = c0 + (idx % 16) * 4;
            vr[u] = j < row1 && c < d ? __ldg(reinterpret_cast<const float4 *>(V + (size_t)j * d + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float acc[4][4] = {};
    if (row0 < row1) fetch(row0);
    for (int j0 = row0; j0 < row1; j0 += kStep) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int idx = tid + u * kThreads;
            if (idx < kStep * TP / 4) *reinterpret_cast<float4 *>(&Ps[idx / (TP / 4)][(idx % (TP / 4)) * 4]) = scaled(kr[u], wt, sc[u]);
        }
#pragma unroll
        for (int u = 0; u < NV; ++u) {
            const int idx = tid + u * kThreads;
            *reinterpret_cast<float4 *>(&Vs[idx / 16][(idx % 16) * 4]) = vr[u];
        }
        __syncthreads();
        if (j0 + kStep < row1) fetch(j0 + kStep);
#pragma unroll
        for (int s = 0; s < kStep / G; ++s) {
            const int jj = s * G + grp;
            const float4 pa = *reinterpret_cast<const float4 *>(&Ps[jj][ty * 4]), vb = *reinterpret_cast<const float4 *>(&Vs[jj][tx * 4]);
            const float pr[4] = {pa.x, pa.y, pa.z, pa.w}, vv[4] = {vb.x, vb.y, vb.z, vb.w};
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(pr[x], vv[y], acc[x][y]);
        }
    }
    chain_next();
    if (G > 1) {
        for (int k = 1; k < G; ++k) {                              // key groups in order
            __syncthreads();
            if (grp == k) {
#pragma unroll
                for (int x = 0; x < 4; ++x)
#pragma unroll
                    for (int y = 0; y < 4; ++y) red[(ty * 4 + x) * kCT + tx * 4 + y] = acc[x][y];
            }
            __syncthreads();
            if (grp == 0) {
#pragma unroll
                for (int x = 0; x < 4; ++x)
#pragma unroll
                    for (int y = 0; y < 4; ++y) acc[x][y] += red[(ty * 4 + x) * kCT + tx * 4 + y];
            }
        }
    }
    const float scale = a.mass2 ? 1.f : (nv > a.skip ? 1.f / (float)(nv - a.skip) : 0.f);
    const int c = c0 + tx * 4;
    if (grp == 0 && c < d) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int t = t0 + ty * 4 + x;
            if (t >= r) continue;
            float4 v = make_float4(acc[x][0], acc[x][1], acc[x][2], acc[x][3]);
            if (a.chunks > 1) {
                __stcg(reinterpret_cast<float4 *>(a.wpart + (((size_t)bh * a.chunks + chunk) * r + t) * d + c), v);
            } else {
                const float f = scale / a.beta[h * r + t];
                *reinterpret_cast<float4 *>(a.Wp + ((size_t)bh * r + t) * d + c) = make_float4(v.x * f, v.y * f, v.z * f, v.w * f);
            }
        }
    }
    if (a.chunks == 1 || !last_of_tile(a.counter + (size_t)bh * gridDim.y + blockIdx.y, a.chunks)) return;
    if (grp == 0 && c < d) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int t = t0 + ty * 4 + x;
            if (t >= r) continue;
            const float *src = a.wpart + ((size_t)bh * a.chunks * r + t) * d + c;
            const float4 s = add_partials(src, (size_t)r * d, a.chunks);
            const float f = scale / a.beta[h * r + t];
            *reinterpret_cast<float4 *>(a.Wp + ((size_t)bh * r + t) * d + c) = make_float4(s.x * f, s.y * f, s.z * f, s.w * f);
        }
    }
}

template <int TS>
__global__ void __launch_bounds__(kThreads, 3)
apply_out_f32_kernel(SweepApplyArgs a)
{
    constexpr int QT = 64, PWD = TS + 1, WW = kCT + 4, NP = QT * TS / 4 / kThreads, NW = TS * kCT / 4 / kThreads < 1 ? 1 : TS * kCT / 4 / kThreads;
    __shared__ float Ps[QT][PWD];                                   // odd pitch: the column reads fall on different banks
    __shared__ __align__(16) float Ws[TS][WW];
    const int bh = blockIdx.z, i0 = blockIdx.x * QT + a.skip, c0 = blockIdx.y * kCT;
    const int n = a.nq, r = a.r, d = a.d, RP = a.RP, tid = threadIdx.x;
    const float *K = a.kt[0] + (size_t)bh * n * RP, *inv = a.inv[0] + (size_t)bh * n, *w = a.w[0] + (size_t)bh * RP;
    const float *W = a.Wp + (size_t)bh * r * d;
    float *O = static_cast<float *>(a.out) + (size_t)bh * n * d;
    const int tx = tid % 16, ty = tid / 16;
    float4 kr[NP], wt[NP], wr[NW];
    float sc[NP];
    chain_wait();
#pragma unroll
    for (int u = 0; u < NP; ++u) {
        const int i = i0 + (tid + u * kThreads) / (TS / 4);
        sc[u] = i < n ? chain_ld(inv + i) : 0.f;
    }
    auto fetch = [&](int tb) {
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int idx = tid + u * kThreads, i = i0 + idx / (TS / 4), t = tb + (idx % (TS / 4)) * 4;
            kr[u] = i < n ? chain_ld4(K + (size_t)i * RP + t) : make_float4(0.f, 0.f, 0.f, 0.f);
            wt[u] = chain_ld4(w + t);
        }
#pragma unroll
        for (int u = 0; u < NW; ++u) {
            const int idx = tid + u * kThreads, t = tb + idx / 16, c = c0 + (idx % 16) * 4;
            wr[u] = idx < TS * 16 && t < r && c < d ? chain_ld4(W + (size_t)t * d + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    float acc[4][4] = {};
    fetch(0);
    for (int tb = 0; tb < r; tb += TS) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int idx = tid + u * kThreads, ii = idx / (TS / 4), t = (idx % (TS / 4)) * 4;
            const float4 p = scaled(kr[u], wt[u], sc[u]);
            Ps[ii][t] = p.x; Ps[ii][t + 1] = p.y; Ps[ii][t + 2] = p.z; Ps[ii][t + 3] = p.w;
        }
#pragma unroll
        for (int u = 0; u < NW; ++u) {
            const int idx = tid + u * kThreads;
            if (idx < TS * 16) *reinterpret_cast<float4 *>(&Ws[idx / 16][(idx % 16) * 4]) = wr[u];
        }
        __syncthreads();
        if (tb + TS < r) fetch(tb + TS);
#pragma unroll
        for (int tt = 0; tt < TS; ++tt) {
            const float4 wb = *reinterpret_cast<const float4 *>(&Ws[tt][tx * 4]);
            const float wv[4] = {wb.x, wb.y, wb.z, wb.w};
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float p = Ps[ty + 16 * x][tt];
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(p, wv[y], acc[x][y]);
            }
        }
    }
    chain_next();
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int i = i0 + ty + 16 * x, c = c0 + tx * 4;
        if (i < n && c < d && LOT_CHECK((size_t)i * d + c + 4 <= (size_t)n * d)) store4(O + (size_t)i * d + c, acc[x]);
    }
}

// ---------------------------------------------------------------------------------------------------------------
template <typename Kern>
static cudaError_t big_smem(Kern kern, size_t bytes)
{
    return bytes > 40 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) : cudaSuccess;
}

template <int TP, int D, int N>
static cudaError_t launch_w(const SweepApplyArgs &a, const SweepApplyArgs *b, cudaStream_t st)
{
    constexpr size_t smem = N * 64 * (TP + 8) * 2 + 64 * (D + 8) * 2;
    auto kern = apply_w_mma_kernel<TP, D, N>;
    cudaError_t e = big_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return chain_launch(kern, dim3(a.chunks, (a.r + TP - 1) / TP, a.B * a.H * (b ? 2 : 1)), kThreads, smem, st, a, b ? *b : a);
}
template <int TP>
static cudaError_t launch_w_d(const SweepApplyArgs &a, const SweepApplyArgs *b, cudaStream_t st)
{
    if (a.d <= 64) return a.terms == 2 ? launch_w<TP, 64, 2>(a, b, st) : launch_w<TP, 64, 3>(a, b, st);
    return a.d <= 128 ? launch_w<TP, 128, 3>(a, b, st) : launch_w<TP, 256, 3>(a, b, st);
}
template <int TS, int D, int N>
static cudaError_t launch_out(const SweepApplyArgs &a, cudaStream_t st)
{
    constexpr size_t smem = N * TS * (D + 8) * 2;
    auto kern = apply_out_mma_kernel<TS, D, N>;
    cudaError_t e = big_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return chain_launch(kern, dim3((a.nq + 127) / 128, a.B * a.H), kThreads, smem, st, a);
}
template <int TS>
static cudaError_t launch_out_d(const SweepApplyArgs &a, cudaStream_t st)
{
    if (a.d <= 64) return a.terms == 2 ? launch_out<TS, 64, 2>(a, st) : launch_out<TS, 64, 3>(a, st);
    return a.d <= 128 ? launch_out<16, 128, 3>(a, st) : launch_out<16, 256, 3>(a, st);
}

} // namespace sweep_apply

cudaError_t launch_sweep_apply_w(const SweepApplyArgs &a, int dtype, cudaStream_t st, const SweepApplyArgs *second)
{
    using namespace sweep_apply;
    if (dtype != 0) return a.RP == 16 ? launch_w_d<16>(a, second, st) : a.RP == 32 ? launch_w_d<32>(a, second, st) : launch_w_d<64>(a, second, st);
    const int cb = (a.d + kCT - 1) / kCT, TP = a.RP < 64 ? a.RP : 64;
    dim3 grid(a.chunks, (a.r + TP - 1) / TP * cb, a.B * a.H);
    return chain_launch(TP == 16 ? apply_w_f32_kernel<16> : TP == 32 ? apply_w_f32_kernel<32> : apply_w_f32_kernel<64>, grid, kThreads, 0, st, a);
}

cudaError_t launch_sweep_apply_out(const SweepApplyArgs &a, int dtype, cudaStream_t st)
{
    using namespace sweep_apply;
    if (dtype != 0) {
        return a.RP == 16 ? launch_out_d<16>(a, st) : launch_out_d<32>(a, st);
    }
    dim3 grid((a.nq + 63) / 64, (a.d + kCT - 1) / kCT, a.B * a.H);
    return chain_launch(a.RP == 16 ? apply_out_f32_kernel<16> : apply_out_f32_kernel<32>, grid, kThreads, 0, st, a);
}

} // namespace lot
