// Last stage of the backward of bf16 tensors (lot_sweep_bwd.cu) up to 64 pivots: the gradient with respect to the similarities is put together
// in shared memory and multiplied at once, dX = dC Z and dZ = dC^T X, both sides in one launch; dC with the reverse steps'
// terms never exists in memory.
//
// Block = one chunk of a problem's rows, 64 at a time: dC_it = dC0_it + K_it sum_k (coef^k_i.x w^k_t - coef^k_i.y f^k_t) in float32, split
// exactly into three bf16 terms (planes) on the way to the tensor cores; Z as three terms too, X as it is; the products of
// total order up to two, small ones first, as in lot_sweep_apply.cu.  Bound by issue (the multiply-adds of the terms, 8 T per four
// entries, the splitting, the products), two blocks an SM in one wave.  Before, one kernel put dC together and four
// multiplied it, five passes over dC.  Whole backward with this kernel and both key-side products in one launch: n = 4096, H = 16,
// r = 64, T = 10 280 -> 252 us (this kernel 57, the five 84), B = 32, H = 3, n = 197, r = 16 82.4 -> 66.7 us (13, the five 38).
#include "lot_chain.cuh"
#include "lot_internal.h"
#include "lot_logits.cuh"
#include "lot_sweep.h"

namespace lot {
namespace grad {

using logits::ldsm4;
using logits::ldsm4_t;
using logits::split;
using logits::smem_addr;
constexpr int kThreads = 256, kRows = 64;

template <int RP, int D> struct Shape {
    static constexpr int PP = (RP + 8) * 2, PX = (D + 8) * 2, PLANE = kRows * PP, ZPLANE = RP * PX;     // pitches: conflict-free ldmatrix
    static constexpr int KS = RP == 64 && D == 128 ? 8 : 16;                                          // reverse steps staged together
    static constexpr int offX = 3 * PLANE, offZ = offX + kRows * PX, offC = offZ + 3 * ZPLANE, offW = offC + 2 * KS * kRows * 8, total = offW + 2 * KS * RP * 4;
};

template <int RP, int D>
__global__ void __launch_bounds__(kThreads, RP == 64 && D == 128 ? 1 : 2)
grad_kernel(const __grid_constant__ SweepGradArgs ga)
{
    typedef Shape<RP, D> Sh;
    constexpr int PT = RP / 16, CG = 8 / PT < D / 16 ? 8 / PT : D / 16, KS = 8 / (PT * CG), NTW = D / 8 / CG;    // dZ: pivot tiles x channels x rows
    constexpr int NP = kRows * RP / 4 / kThreads, NX = kRows * D / 8 / kThreads, NZ = RP * D / 4 / kThreads;
    extern __shared__ __align__(128) uint8_t sm[];
    uint8_t *sP = sm, *sX = sm + Sh::offX, *sZ = sm + Sh::offZ;
    float2 *sc = reinterpret_cast<float2 *>(sm + Sh::offC);
    float *sw = reinterpret_cast<float *>(sm + Sh::offW), *sf = sw + Sh::KS * RP;
    const SweepBwdArgs &a = ga.b;
    const SweepArgs &s = a.s;
    const int p = blockIdx.y, slice = p >> 1, side = (p & 1) ^ 1, h = slice % s.H, n = s.n[side], r = s.r, d = s.d, NP2 = 2 * s.B * s.H;
    int nv = n;
    if (side == 1 && s.key_len != nullptr) nv = min(max(__ldg(s.key_len + slice / s.H), 0), n);
    const int chunk = blockIdx.x, row0 = chunk * ga.rows, row1 = min(row0 + ga.rows, n);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3, mi = lane >> 3;
    const int pt = warp % PT, cg = (warp / PT) % CG, ks = warp / (PT * CG);      // dZ
    const int rt = warp & 3, ch = warp >> 2;                                     // dX: 16 rows, half of the channels
    // the pivots depend on no earlier kernel
    const float *z = s.z + (size_t)h * r * d;
#pragma unroll
    for (int u = 0; u < NZ; ++u) {
        const int idx = tid + u * kThreads, t = idx / (D / 4), c = (idx % (D / 4)) * 4;
        const float4 v = t < r && c < d ? __ldg(reinterpret_cast<const float4 *>(z + (size_t)t * d + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t x[3], y[3];
        split<3>(v.x, v.y, x);
        split<3>(v.z, v.w, y);
#pragma unroll
        for (int i = 0; i < 3; ++i) *reinterpret_cast<uint2 *>(sZ + i * Sh::ZPLANE + t * Sh::PX + c * 2) = make_uint2(x[i], y[i]);
    }
    const float *K = s.kt[side] + (size_t)slice * n * RP, *dC = a.dC[side] + (size_t)slice * n * RP;
    const __nv_bfloat16 *X = static_cast<const __nv_bfloat16 *>(s.x[side]) + (size_t)slice * n * d;
    const float2 *coef = a.coef + (size_t)p * a.T * n;
    chain_wait();
    // A wide problem's dC is complete, and its kernel is not to be read: the reverse steps left exponents in place of the rows that were not in
    // shared memory, -infinity in the columns behind r.
    const int T = nv == 0 || *reinterpret_cast<const volatile int *>(s.wide + p) != 0 ? 0 : a.T;
    __nv_bfloat16 *dX = static_cast<__nv_bfloat16 *>(ga.dx[side]) + (size_t)slice * n * d;

    float4 kr[NP], dr[NP];
    uint4 xr[NX];
    auto fetch = [&](int j0) {
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int idx = tid + u * kThreads, j = j0 + idx / (RP / 4), t = (idx % (RP / 4)) * 4;
            const bool in = j < nv && j < row1;
            kr[u] = in && T > 0 ? chain_ld4(K + (size_t)j * RP + t) : make_float4(0.f, 0.f, 0.f, 0.f);
            dr[u] = in ? chain_ld4(dC + (size_t)j * RP + t) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < NX; ++u) {
            const int idx = tid + u * kThreads, j = j0 + idx / (D / 8), c = (idx % (D / 8)) * 8;
            xr[u] = j < nv && j < row1 && c < d ? __ldg(reinterpret_cast<const uint4 *>(X + (size_t)j * d + c)) : make_uint4(0, 0, 0, 0);
        }
    };
    // the first KS steps' coefficients of 64 rows, into the set of that turn
    auto fetch_coef = [&](int j0, int T, int turn) {
        const int kn = min(Sh::KS, T);
        for (int idx = tid; idx < kn * kRows; idx += kThreads) {
            const int k = idx / kRows, j = j0 + idx % kRows;
            const bool in = j < nv && j < row1;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_addr(sc + (turn & 1) * (Sh::KS * kRows) + idx)),
                         "l"(coef + (size_t)k * n + (in ? j : 0)), "r"(in ? 8 : 0) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[NTW][4] = {};
    if (row0 < row1) {
        fetch(row0);
        fetch_coef(row0, T, 0);
    }
    for (int j0 = row0, turn = 0; j0 < row1; j0 += kRows, ++turn) {
        float4 e[NP];
        float2 *cc = sc + (turn & 1) * (Sh::KS * kRows);
#pragma unroll
        for (int u = 0; u < NP; ++u) e[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k0 = 0; k0 < T; k0 += Sh::KS) {
            const int kn = min(Sh::KS, T - k0);
            if (k0 == 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();                                       // the last step's products, or these buffers, are done with
            if (k0 > 0)
                for (int idx = tid; idx < kn * kRows; idx += kThreads) {
                    const int k = idx / kRows, i = idx % kRows;
                    cc[idx] = j0 + i < nv && j0 + i < row1 ? chain_ld2(reinterpret_cast<const float *>(coef + (size_t)(k0 + k) * n + j0 + i)) : make_float2(0.f, 0.f);
                }
            if (T > Sh::KS || j0 == row0)
                for (int idx = tid; idx < kn * RP; idx += kThreads) {
                    const size_t o = ((size_t)(k0 + idx / RP) * NP2 + p) * RP + idx % RP;
                    sw[idx] = chain_ld(s.hist + o);
                    sf[idx] = chain_ld(a.fk + o);
                }
            if (T > Sh::KS || j0 == row0) __syncthreads();
#pragma unroll 4
            for (int k = 0; k < kn; ++k) {
                const int t = (tid % (RP / 4)) * 4;                // kThreads is a multiple of RP / 4
                const float4 w = *reinterpret_cast<const float4 *>(sw + k * RP + t), f = *reinterpret_cast<const float4 *>(sf + k * RP + t);
#pragma unroll
                for (int u = 0; u < NP; ++u) {
                    const float2 c = cc[k * kRows + (tid + u * kThreads) / (RP / 4)];
                    e[u].x = fmaf(c.x, w.x, fmaf(-c.y, f.x, e[u].x));
                    e[u].y = fmaf(c.x, w.y, fmaf(-c.y, f.y, e[u].y));
                    e[u].z = fmaf(c.x, w.z, fmaf(-c.y, f.z, e[u].z));
                    e[u].w = fmaf(c.x, w.w, fmaf(-c.y, f.w, e[u].w));
                }
            }
        }
        if (T == 0) __syncthreads();
#pragma unroll
        for (int u = 0; u < NP; ++u) {
            const int idx = tid + u * kThreads, j = idx / (RP / 4), t = (idx % (RP / 4)) * 4;
            uint32_t x[3], y[3];
            split<3>(fmaf(kr[u].x, e[u].x, dr[u].x), fmaf(kr[u].y, e[u].y, dr[u].y), x);
            split<3>(fmaf(kr[u].z, e[u].z, dr[u].z), fmaf(kr[u].w, e[u].w, dr[u].w), y);
#pragma unroll
            for (int i = 0; i < 3; ++i) *reinterpret_cast<uint2 *>(sP + i * Sh::PLANE + j * Sh::PP + t * 2) = make_uint2(x[i], y[i]);
        }
#pragma unroll
        for (int u = 0; u < NX; ++u) {
            const int idx = tid + u * kThreads;
            *reinterpret_cast<uint4 *>(sX + (idx / (D / 8)) * Sh::PX + (idx % (D / 8)) * 16) = xr[u];
        }
        __syncthreads();
        if (j0 + kRows < row1) {
            fetch(j0 + kRows);
            fetch_coef(j0 + kRows, T, turn + 1);
        }
        // dZ += dC^T X
#pragma unroll
        for (int st = 0; st < kRows / 16 / KS; ++st) {
            const int j = (ks * (kRows / 16 / KS) + st) * 16;
            uint32_t af[3][4];
#pragma unroll
            for (int i = 0; i < 3; ++i)
                ldsm4_t(af[i], smem_addr(sP) + i * Sh::PLANE + (j + (lane & 7) + (mi >> 1) * 8) * Sh::PP + (pt * 16 + (mi & 1) * 8) * 2);
#pragma unroll
            for (int nt = 0; nt < NTW; nt += 2) {
                uint32_t bf[4];
                ldsm4_t(bf, smem_addr(sX) + (j + (lane & 7) + (mi & 1) * 8) * Sh::PX + (cg * NTW * 8 + nt * 8 + (mi >> 1) * 8) * 2);
#pragma unroll
                for (int i = 2; i >= 0; --i) {
                    logits::mma_bf16(acc[nt], af[i], bf[0], bf[1]);
                    logits::mma_bf16(acc[nt + 1], af[i], bf[2], bf[3]);
                }
            }
        }
        // dX = dC Z
        float o[D / 16][4] = {};
#pragma unroll
        for (int k = 0; k < RP / 16; ++k) {
            uint32_t af[3][4];
#pragma unroll
            for (int i = 0; i < 3; ++i) ldsm4(af[i], smem_addr(sP) + i * Sh::PLANE + (rt * 16 + (lane & 15)) * Sh::PP + (k * 16 + (lane >> 4) * 8) * 2);
#pragma unroll
            for (int cp = 0; cp < D / 32; ++cp) {
                uint32_t bf[3][4];
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    ldsm4_t(bf[i], smem_addr(sZ) + i * Sh::ZPLANE + (k * 16 + (lane & 7) + (mi & 1) * 8) * Sh::PX + (ch * (D / 2) + cp * 16 + (mi >> 1) * 8) * 2);
#pragma unroll
                for (int ord = 2; ord >= 0; --ord)
#pragma unroll
                    for (int i = 0; i <= ord; ++i) {
                        logits::mma_bf16(o[2 * cp], af[i], bf[ord - i][0], bf[ord - i][1]);
                        logits::mma_bf16(o[2 * cp + 1], af[i], bf[ord - i][2], bf[ord - i][3]);
                    }
            }
        }
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int j = j0 + rt * 16 + g + 8 * hh;
            if (j >= row1) continue;
#pragma unroll
            for (int t = 0; t < D / 16; ++t) {
                const int c = ch * (D / 2) + 8 * t + 2 * q;
                if (c < d) *reinterpret_cast<__nv_bfloat162 *>(dX + (size_t)j * d + c) = __floats2bfloat162_rn(o[t][2 * hh], o[t][2 * hh + 1]);
            }
        }
    }
    chain_next();
    if (KS > 1) {                                                  // halves of the rows
        float *red = reinterpret_cast<float *>(sm);
        __syncthreads();
        if (ks > 0) {
#pragma unroll
            for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
                for (int v = 0; v < 4; ++v) red[(((ks - 1) * PT * CG + warp % (PT * CG)) * NTW * 4 + nt * 4 + v) * 32 + lane] = acc[nt][v];
        }
        __syncthreads();
        if (ks > 0) return;
        for (int k2 = 1; k2 < KS; ++k2)
#pragma unroll
            for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
                for (int v = 0; v < 4; ++v) acc[nt][v] += red[(((k2 - 1) * PT * CG + warp) * NTW * 4 + nt * 4 + v) * 32 + lane];
    }
    float *part = ga.part[side] + ((size_t)slice * ga.chunks + chunk) * r * d;
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            const int t = pt * 16 + g + 8 * hh, c = cg * NTW * 8 + nt * 8 + 2 * q;
            if (t < r && c < d) *reinterpret_cast<float2 *>(part + (size_t)t * d + c) = make_float2(acc[nt][2 * hh], acc[nt][2 * hh + 1]);
        }
}

template <int RP, int D> static cudaError_t launch_t(const SweepGradArgs &a, cudaStream_t st)
{
    constexpr size_t smem = Shape<RP, D>::total;
    if (smem > 40 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(grad_kernel<RP, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return chain_launch(grad_kernel<RP, D>, dim3(a.chunks, 2 * a.b.s.B * a.b.s.H), kThreads, smem, st, a);
}

} // namespace grad

// One wave of blocks, two to an SM, in whole steps.
int sweep_grad_chunks(int BH, int n)
{
    const int steps = (n + grad::kRows - 1) / grad::kRows, want = device_sm_count() / (BH > 0 ? BH : 1);
    const int per = (steps + (want > 0 ? want : 1) - 1) / (want > 0 ? want : 1);
    return (steps + per - 1) / per;
}

bool sweep_grad_supported(int r, int d) { return r <= 64 && d <= 128; }

cudaError_t launch_sweep_grad(int RP, const SweepGradArgs &a, cudaStream_t st)
{
    using namespace grad;
    const bool wide = a.b.s.d > 64;
    if (RP == 16) return wide ? launch_t<16, 128>(a, st) : launch_t<16, 64>(a, st);
    if (RP == 32) return wide ? launch_t<32, 128>(a, st) : launch_t<32, 64>(a, st);
    return wide ? launch_t<64, 128>(a, st) : launch_t<64, 64>(a, st);
}

} // namespace lot
