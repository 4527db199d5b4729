// Backward of bf16 tensors on the stored Gibbs kernel (Section "Learning"; what is differentiated: lot_backward.cu).
//
// In the scaling form the plan of iteration k is R^k_it = K_it w^k_t / s^k_i, and with f^k_t = w^k_t gamma_t / beta_t (the
// weights after the pivot update being reversed) the reverse of one iteration reads
//     s_i = sum_t K_it w_t,  u_i = sum_t K_it f_t,  rho_i = u_i / s_i,      gamma'_t = m w_t sum_i K_it u_i / s_i^2,
//     dC_it += K_it (w_t m u_i / s_i^2 - f_t m / s_i):
// a read-only pass like the forward's, and a rank-two term on top of K.  So the reverse iterations only keep two numbers
// per row and two per column, and the gradient with respect to the similarities is put together once at the end
// (assemble_kernel, or up to 64 pivots lot_sweep_grad.cu) instead of being read and written in every iteration.
// Problems whose potentials ranged over more than the kernel's window are reversed step by step on rebuilt exponents.
#include "lot_chain.cuh"
#include "lot_sweep_core.cuh"

#include <mutex>

namespace lot {
namespace sweep {

// ---------------------------------------------------------------------------------------------------------------
// Closing update and read-out: dR = g . wmat^T, rho_i = sum_t R_it dR_it, dC_it = R_it (dR_it - rho_i) / eps and its column
// sums.  Block = 128 rows, a warp's rows stay in its accumulators (as in lot_build.cu).
// ---------------------------------------------------------------------------------------------------------------
template <int RP>
__global__ void __launch_bounds__(256, RP <= 64 ? 2 : 1)
close_kernel(const __grid_constant__ SweepBwdArgs a)
{
    extern __shared__ __align__(128) uint8_t stage[];
    __shared__ float sw[RP];
    __shared__ float red[8][RP];
    typedef logits::Logits<__nv_bfloat16, RP, 16, 256> Lg;
    const SweepArgs &s = a.s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3, r = s.r, d = s.d;
    const int p = blockIdx.x / a.tiles, tile = blockIdx.x % a.tiles, slice = p >> 1, side = (p & 1) ^ 1, n = s.n[side];
    int nv = n;
    if (side == 1 && s.key_len != nullptr) nv = min(max(__ldg(s.key_len + slice / s.H), 0), n);
    const int w0 = tile * 128 + warp * 16, wrows = min(max(nv - w0, 0), 16);
    float *gp = a.gpart + ((size_t)p * a.tiles + tile) * RP;
    chain_wait();
    if (tile * 128 >= nv) {
        if (threadIdx.x < RP) gp[threadIdx.x] = 0.f;
        return;
    }
    if (threadIdx.x < RP) sw[threadIdx.x] = s.w[side][(size_t)slice * RP + threadIdx.x];
    Lg lg;
    lg.run(static_cast<const __nv_bfloat16 *>(a.g[side]) + ((size_t)slice * n + w0) * d, wrows, d, a.wmat[side] + (size_t)slice * r * d, r,
           stage, lane);
    const float *kt = s.kt[side] + ((size_t)slice * n + w0) * RP, *inv = s.inv[side] + (size_t)slice * n + w0;
    float *dC = a.dC[side] + ((size_t)slice * n + w0) * RP;
    const float inv_eps = (float)(1.0 / a.eps);
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        const int i = g + 8 * hh;
        const bool ok = i < wrows;
        const float iv = ok ? inv[i] : 0.f;
        float rho = 0.f;
#pragma unroll
        for (int j = 0; j < RP / 8; ++j) {
            const int t = 8 * j + 2 * q;
            const float2 k = ok ? *reinterpret_cast<const float2 *>(kt + (size_t)i * RP + t) : make_float2(0.f, 0.f);
            rho = fmaf(k.x * (sw[t] * iv), lg.at(j, hh, 0), rho);
            rho = fmaf(k.y * (sw[t + 1] * iv), lg.at(j, hh, 1), rho);
        }
        rho += __shfl_xor_sync(0xffffffffu, rho, 1);
        rho += __shfl_xor_sync(0xffffffffu, rho, 2);
#pragma unroll
        for (int j = 0; j < RP / 8; ++j) {
            const int t = 8 * j + 2 * q;
            const float2 k = ok ? *reinterpret_cast<const float2 *>(kt + (size_t)i * RP + t) : make_float2(0.f, 0.f);
            float2 v;
            v.x = k.x * (sw[t] * iv) * (lg.at(j, hh, 0) - rho) * inv_eps;
            v.y = k.y * (sw[t + 1] * iv) * (lg.at(j, hh, 1) - rho) * inv_eps;
            if (ok) *reinterpret_cast<float2 *>(dC + (size_t)i * RP + t) = v;
            lg.at(j, hh, 0) = ok ? v.x : 0.f;
            lg.at(j, hh, 1) = ok ? v.y : 0.f;
        }
    }
    chain_next();
#pragma unroll
    for (int j = 0; j < RP / 8; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float c = lg.at(j, 0, e) + lg.at(j, 1, e);
            c += __shfl_xor_sync(0xffffffffu, c, 4);
            c += __shfl_xor_sync(0xffffffffu, c, 8);
            c += __shfl_xor_sync(0xffffffffu, c, 16);
            if (g == 0) red[warp][8 * j + 2 * q + e] = c;
        }
    __syncthreads();
    if (threadIdx.x < RP) {
        float c = red[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < 8; ++w) c += red[w][threadIdx.x];
        gp[threadIdx.x] = c;
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Reverse iterations
// ---------------------------------------------------------------------------------------------------------------
// One reverse pass over the block's rows: column sums of K u / s^2, row coefficients to coef.
template <int RP, int CPL, int THREADS, bool TENSOR>
__device__ __forceinline__ void reverse_pass(const Lane<RP, CPL> &L, const Share &R, const u64 (&w)[CPL / 2], const u64 (&f)[CPL / 2],
                                             u64 (&acc)[CPL / 2], float mass, float2 *coef)
{
    typedef Lay<RP, CPL> Y;
    constexpr int STEP = (THREADS / 32) * Y::RPW;
#pragma unroll
    for (int j = 0; j < CPL / 2; ++j) acc[j] = 0;
    auto one = [&](const Row<CPL> &k, int i, int end) {
        u64 s2 = 0, u2 = 0;
#pragma unroll
        for (int j = 0; j < CPL / 2; ++j) { s2 = fma_f2(k.k[j], w[j], s2); u2 = fma_f2(k.k[j], f[j], u2); }
        float a, b, s, u;
        unpack_f2(s2, a, b);
        s = a + b;
        unpack_f2(u2, a, b);
        u = a + b;
#pragma unroll
        for (int off = Y::LPR / 2; off > 0; off >>= 1) {
            s += __shfl_xor_sync(0xffffffffu, s, off);
            u += __shfl_xor_sync(0xffffffffu, u, off);
        }
        const float inv = rcp(fmaxf(s, 1e-37f)), x = u * inv * inv;
        const u64 xx = pack_f2(x, x);
#pragma unroll
        for (int j = 0; j < CPL / 2; ++j) acc[j] = fma_f2(k.k[j], xx, acc[j]);
        if (L.cl == 0 && i < end) coef[i] = make_float2(mass * x, mass * inv);
    };
    for (int st = 0; st < R.steps; ++st) {
        Row<CPL> k;
#pragma unroll
        for (int v = 0; v < Y::NV; ++v) lds2(k.k[2 * v], k.k[2 * v + 1], L.template chunk<TENSOR && RP <= 32>(st * (STEP * RP * 4), v));
        one(k, L.i0 + st * STEP, R.ns);
    }
    const int on_chip = TENSOR ? R.ns + R.nt : R.ns;
#pragma unroll 1
    for (int ts = 0; TENSOR && ts < R.tsteps; ++ts) {
        u64 k2[8];
        tensor_load<16>(k2, L.t + ts * CPL);
        tensor_settle<16>(k2);
        Row<CPL> k;
#pragma unroll
        for (int j = 0; j < CPL / 2; ++j) k.k[j] = k2[j];
        one(k, R.ns + L.i0 + ts * STEP, on_chip);
    }
    if (on_chip < R.nrows)
        for (int i = on_chip + L.i0; i - L.i0 < R.nrows; i += STEP) {
            Row<CPL> k;
#pragma unroll
            for (int v = 0; v < Y::NV; ++v) {
                const ulonglong2 t = i < R.nrows ? __ldcg(reinterpret_cast<const ulonglong2 *>(R.g + (size_t)i * RP) + v * Y::LPR + L.cl)
                                                 : make_ulonglong2(0, 0);
                k.k[2 * v] = t.x;
                k.k[2 * v + 1] = t.y;
            }
            one(k, i, R.nrows);
        }
}

// The reverse iterations of a problem whose kept weights leave float32's range: exponents around the potentials of every
// iteration, dC updated in place.  gam: thread t's gradient with respect to the last potentials.
template <int RP, int CPL, int THREADS, bool GROUP>
__device__ __noinline__ unsigned reverse_wide(const SweepBwdArgs *ap, int p, int group, int c, unsigned seq, float gam)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    typedef Lay<RP, CPL> Y;
    const SweepArgs &s = ap->s;
    const Shared S = carve<__nv_bfloat16, RP, THREADS>(smem, s.srows);
    Share R;
    const Problem P = locate<RP, CPL, THREADS>(s, p, c, R);
    const __nv_bfloat16 *x = static_cast<const __nv_bfloat16 *>(s.x[P.side]) + ((size_t)P.slice * P.n + P.row0) * s.d;
    const float *z = s.z + (size_t)P.h * s.r * s.d;
    float *dC = ap->dC[P.side] + ((size_t)P.slice * P.n + P.row0) * RP;
    const int tid = threadIdx.x, r = s.r, NP = 2 * s.B * s.H;
    const int lane = tid & 31, warp = tid >> 5, sub = lane / Y::LPR, cl = lane % Y::LPR;
    constexpr int STEP = (THREADS / 32) * Y::RPW;
    const float mass = 1.f / (float)P.nv, beta = tid < r ? __ldg(s.beta + P.h * r + tid) : 1.f;
    float db = 0.f;
    for (int it = ap->T; it >= 1; --it) {
        __syncthreads();
        if (tid < RP) {
            const double *hg = s.hist_g + (size_t)p * RP + tid;
            const double ga = tid < r ? hg[(size_t)(it - 1) * NP * RP] : 0.0, gb = tid < r ? hg[(size_t)it * NP * RP] : 0.0;
            S.gref[tid] = ga;
            S.w[tid] = tid < r ? (float)(gb - ga - log2((double)beta)) : neg_inf();
            S.tgt[tid] = tid < r ? gam : 0.f;
            db += (float)ap->eps * gam / beta;
        }
        __syncthreads();
        build<__nv_bfloat16, RP, CPL, THREADS, true>(S, R, x, z, s.d, r, s.scale);
        float v[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) v[k] = 0.f;
        for (int base = warp * Y::RPW; base < R.nrows; base += STEP) {
            const int i = base + sub;
            const bool ok = i < R.nrows;
            float e[CPL], sum = 0.f, rho = 0.f;
#pragma unroll
            for (int u = 0; u < Y::NV; ++u) {
                const float4 t = ok ? *chunk_ptr<RP, CPL>(S, R, i, u * Y::LPR + cl) : make_float4(0.f, 0.f, 0.f, 0.f);
                e[4 * u] = t.x; e[4 * u + 1] = t.y; e[4 * u + 2] = t.z; e[4 * u + 3] = t.w;
            }
#pragma unroll
            for (int k = 0; k < CPL; ++k) sum += ex2(e[k]);
            sum = group_sum(sum, Y::LPR);
            const float lgs = lg2(sum);
            float qg[CPL];
#pragma unroll
            for (int k = 0; k < CPL; ++k) {
                const int t = ((k >> 2) * Y::LPR + cl) * 4 + (k & 3);
                qg[k] = ex2(e[k] - lgs + S.w[t]) * S.tgt[t];
                rho += qg[k];
            }
            rho = group_sum(rho, Y::LPR);
#pragma unroll
            for (int u = 0; u < Y::NV; ++u) {
                float4 *dp = reinterpret_cast<float4 *>(dC + (size_t)i * RP) + u * Y::LPR + cl;
                float4 o = ok ? *dp : make_float4(0.f, 0.f, 0.f, 0.f);
                float m[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    m[k] = mass * ex2(e[4 * u + k] - lgs) * rho;
                    if (ok) v[4 * u + k] += m[k];
                }
                o.x += m[0] - mass * qg[4 * u];
                o.y += m[1] - mass * qg[4 * u + 1];
                o.z += m[2] - mass * qg[4 * u + 2];
                o.w += m[3] - mass * qg[4 * u + 3];
                if (ok) *dp = o;
            }
        }
        gam = block_columns<RP, CPL, THREADS, false>(S, v);
        if (GROUP) gam = group_columns<RP, THREADS, false>(s, S, gam, group, c, seq);
    }
    if (c == 0 && tid < r) ap->dbeta_acc[(size_t)p * RP + tid] = db;
    return seq;
}

template <int RP, int CPL, int THREADS, bool GROUP, bool TENSOR>
__global__ void __launch_bounds__(THREADS, max_blocks(CPL, THREADS))
reverse_kernel(const __grid_constant__ SweepBwdArgs a)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    typedef Lay<RP, CPL> Y;
    const SweepArgs &s = a.s;
    const int tid = threadIdx.x, group = GROUP ? blockIdx.x / s.C : blockIdx.x, c = GROUP ? blockIdx.x % s.C : 0;
    const int NP = 2 * s.B * s.H, r = s.r;
    unsigned seq = s.seq0;
    const Shared S = carve<__nv_bfloat16, RP, THREADS>(smem, s.srows);
    if (tid == 0) S.flag[0] = 0;
    if (GROUP) open_exchange<RP>(s, S);
    if (TENSOR) open_tensor(S, s.tcols);
    chain_wait();

    for (int p = group; p < NP; p += s.groups) {
        Share R;
        const Problem P = locate<RP, CPL, THREADS>(s, p, c, R);
        if (P.nv <= 0) {
            if (c == 0 && tid < RP) a.dbeta_acc[(size_t)p * RP + tid] = 0.f;
            continue;
        }
        float gam = 0.f;
        if (tid < RP)
            for (int k = 0; k < a.tiles; ++k) gam += a.gpart[((size_t)p * a.tiles + k) * RP + tid];
        const bool wide = s.wide[p] != 0;
        __syncthreads();
        if (wide) {
            seq = reverse_wide<RP, CPL, THREADS, GROUP>(&a, p, group, c, seq, gam);
            continue;
        }
        load_rows<RP, CPL, THREADS>(S, R);
        if constexpr (TENSOR) load_tensor_rows<RP, CPL, THREADS>(S, R, s.tcols);
        const float *hw = s.hist + (size_t)p * RP + (tid < RP ? tid : 0);
        const size_t hstep = (size_t)NP * RP;
        const float beta = tid < r ? __ldg(s.beta + P.h * r + tid) : 1.f, mass = 1.f / (float)P.nv;
        float wb = hw[(size_t)a.T * hstep], wa = a.T > 0 ? hw[(size_t)(a.T - 1) * hstep] : 0.f, db = 0.f;
        const Lane<RP, CPL> L = make_lane<RP, CPL, THREADS>(S, s.tcols);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        const uint32_t f_addr = smem_addr(S.tgt) + L.cl * 16;
        float2 *coef = a.coef + (size_t)p * a.T * P.n + P.row0;
        for (int it = a.T; it >= 1; --it) {
            if (tid < RP) {
                const float f = tid < r ? wb * gam / beta : 0.f;
                db += (float)a.eps * gam / beta;
                S.w[tid] = tid < r ? wa : 0.f;
                S.tgt[tid] = f;
                if (c == 0) a.fk[((size_t)(it - 1) * NP + p) * RP + tid] = f;
            }
            __syncthreads();
            u64 w[CPL / 2], f[CPL / 2], acc[CPL / 2];
            load_weights<RP, CPL>(L, w);
#pragma unroll
            for (int v = 0; v < CPL / 4; ++v) lds2(f[2 * v], f[2 * v + 1], f_addr + v * (Y::LPR * 16));
            const float wnext = it >= 2 ? hw[(size_t)(it - 2) * hstep] : 0.f;
            reverse_pass<RP, CPL, THREADS, TENSOR>(L, R, w, f, acc, mass, coef + (size_t)(it - 1) * P.n);
            float v[CPL];
#pragma unroll
            for (int j = 0; j < CPL / 2; ++j) unpack_f2(acc[j], v[2 * j], v[2 * j + 1]);
            float tot = block_columns<RP, CPL, THREADS, false>(S, v);
            if (GROUP) tot = group_columns<RP, THREADS, false>(s, S, tot, group, c, seq);
            gam = mass * wa * tot;
            wb = wa;
            wa = wnext;
        }
        if (p + s.groups >= NP) chain_next();
        if (c == 0 && tid < r) a.dbeta_acc[(size_t)p * RP + tid] = db;
        __syncthreads();
    }
    if (TENSOR) close_tensor(S, s.tcols);
    if (GROUP) close_exchange(s);
}

// ---------------------------------------------------------------------------------------------------------------
// More than 64 pivots or 128 channels: dC_it += K_it sum_k (coef^k_i.x w^k_t - coef^k_i.y f^k_t), 4 rows x 4 columns per thread, the
// coefficients of KS iterations at a time in shared memory.
// ---------------------------------------------------------------------------------------------------------------
template <int RP>
__global__ void __launch_bounds__(256)
assemble_kernel(const __grid_constant__ SweepBwdArgs a)
{
    constexpr int CT = RP < 64 ? RP : 64, TC = CT / 4, ROWS = 256 / TC * 4, KS = ROWS == 64 ? 16 : ROWS == 128 ? 8 : 4;
    __shared__ __align__(16) float2 sc[KS][ROWS + 1];
    __shared__ __align__(16) float sw[KS][CT], sf[KS][CT];
    const SweepArgs &s = a.s;
    const int p = blockIdx.z, slice = p >> 1, side = (p & 1) ^ 1, n = s.n[side], NP = 2 * s.B * s.H;
    int nv = n;
    if (side == 1 && s.key_len != nullptr) nv = min(max(__ldg(s.key_len + slice / s.H), 0), n);
    const int i0 = blockIdx.x * ROWS, t0 = blockIdx.y * CT, tid = threadIdx.x;
    chain_wait();
    if (i0 >= nv || s.wide[p] != 0) return;
    const int tx = tid % TC, ty = tid / TC;
    const float2 *coef = a.coef + (size_t)p * a.T * n + i0;
    float acc[4][4] = {};
    for (int k0 = 0; k0 < a.T; k0 += KS) {
        __syncthreads();
        for (int idx = tid; idx < KS * ROWS; idx += 256) {
            const int k = idx / ROWS, i = idx % ROWS;
            sc[k][i] = k0 + k < a.T && i0 + i < nv ? coef[(size_t)(k0 + k) * n + i] : make_float2(0.f, 0.f);
        }
        for (int idx = tid; idx < KS * CT; idx += 256) {
            const int k = idx / CT, t = idx % CT;
            const size_t o = ((size_t)(k0 + k) * NP + p) * RP + t0 + t;
            sw[k][t] = k0 + k < a.T ? s.hist[o] : 0.f;
            sf[k][t] = k0 + k < a.T ? a.fk[o] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const float4 w = *reinterpret_cast<const float4 *>(&sw[k][tx * 4]), f = *reinterpret_cast<const float4 *>(&sf[k][tx * 4]);
            const float wv[4] = {w.x, w.y, w.z, w.w}, fv[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float2 cc = sc[k][ty + x * (256 / TC)];
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(cc.x, wv[y], fmaf(-cc.y, fv[y], acc[x][y]));
            }
        }
    }
    chain_next();
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int i = i0 + ty + x * (256 / TC);
        if (i >= nv) continue;
        const size_t o = ((size_t)slice * n + i) * RP + t0 + tx * 4;
        const float4 k = *reinterpret_cast<const float4 *>(s.kt[side] + o);
        float4 v = *reinterpret_cast<const float4 *>(a.dC[side] + o);
        v.x = fmaf(k.x, acc[x][0], v.x); v.y = fmaf(k.y, acc[x][1], v.y); v.z = fmaf(k.z, acc[x][2], v.z); v.w = fmaf(k.w, acc[x][3], v.w);
        *reinterpret_cast<float4 *>(a.dC[side] + o) = v;
    }
}

__global__ void merge_kernel(const float *part_q, const float *part_k, const float *dbeta_direct, const float *dbeta_acc, float *dz, float *dbeta, int B, int H, int d,
                             int r, int RP, int chunks, bool add)
{
    // eight threads an element, each a share of the partials (of the batch rows for beta), requested eight at a time: bound by
    // latency, 12 us at B = 32, H = 3, r = 16, d = 64 when one thread went through the batch rows of beta
    constexpr int W = 8;
    const size_t per = (size_t)r * d, idx = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) / W;
    const int part = threadIdx.x % W;
    chain_wait();
    float sum = 0.f, bsum = 0.f;
    if (idx < (size_t)H * per) {
        const int h = (int)(idx / per), all = B * chunks, j0 = (int)((long long)all * part / W), j1 = (int)((long long)all * (part + 1) / W);
        const size_t e = idx % per;
#pragma unroll 8
        for (int j = j0; j < j1; ++j) {
            const int b = j / chunks, c = j - b * chunks;
            const size_t o = (((size_t)b * H + h) * chunks + c) * per + e;
            sum += part_q[o] + part_k[o];
        }
    }
    if (idx < (size_t)H * r) {
        const int h = (int)(idx / r), t = (int)(idx % r), b1 = (int)((long long)B * (part + 1) / W);
#pragma unroll 4
        for (int b = (int)((long long)B * part / W); b < b1; ++b) {
            const size_t sl = (size_t)b * H + h;
            bsum += dbeta_direct[sl * r + t] + dbeta_acc[(2 * sl) * RP + t] + dbeta_acc[(2 * sl + 1) * RP + t];
        }
    }
#pragma unroll
    for (int off = 1; off < W; off <<= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, off);
        bsum += __shfl_xor_sync(0xffffffffu, bsum, off);
    }
    if (part == 0 && idx < (size_t)H * per) dz[idx] = add ? dz[idx] + sum : sum;
    if (part == 0 && idx < (size_t)H * r) dbeta[idx] = add ? dbeta[idx] + bsum : bsum;
}

// ---------------------------------------------------------------------------------------------------------------
template <typename Kern> static cudaError_t allow_smem(Kern kern, size_t bytes)
{
    return bytes > 40 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) : cudaSuccess;
}

template <int RP> static cudaError_t close_t(const SweepBwdArgs &a, cudaStream_t st)
{
    constexpr size_t smem = logits::stage_bytes<__nv_bfloat16>(RP);
    cudaError_t e = allow_smem(close_kernel<RP>, smem);
    if (e != cudaSuccess) return e;
    return chain_launch(close_kernel<RP>, dim3((unsigned)(2 * a.s.B * a.s.H * a.tiles)), 256, smem, st, a);
}
template <int RP> static cudaError_t assemble_t(const SweepBwdArgs &a, cudaStream_t st)
{
    constexpr int CT = RP < 64 ? RP : 64, ROWS = 256 / (CT / 4) * 4;
    return chain_launch(assemble_kernel<RP>, dim3((a.s.n[0] + ROWS - 1) / ROWS, RP / CT, 2 * a.s.B * a.s.H), 256, 0, st, a);
}
template <int RP, bool GROUP, bool TENSOR> static cudaError_t reverse_g(const SweepPlan &P, const SweepBwdArgs &a, cudaStream_t st)
{
    constexpr int THREADS = TENSOR ? kTensorThreads : 256;
    auto kern = reverse_kernel<RP, TENSOR ? kTensorLane : wide_cols(RP), THREADS, GROUP, TENSOR>;
    if (P.tcols != 0 && P.smem < kAloneSmem) return cudaErrorInvalidConfiguration;
    cudaError_t e = allow_smem(kern, P.smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(P.groups * P.C));
    if (P.chained) return chain_launch(kern, grid, THREADS, P.smem, P.K, st, a);
    if (P.C == P.K) return cluster_launch(kern, grid, THREADS, P.smem, P.K, st, a);
    return group_launch(kern, grid, THREADS, P.smem, P.K, st, a);
}
template <int RP> static cudaError_t reverse_t(const SweepPlan &P, const SweepBwdArgs &a, cudaStream_t st)
{
    if (P.C > 1) return P.threads == kTensorThreads ? reverse_g<RP, true, true>(P, a, st) : reverse_g<RP, true, false>(P, a, st);
    return P.threads == kTensorThreads ? reverse_g<RP, false, true>(P, a, st) : reverse_g<RP, false, false>(P, a, st);
}

} // namespace sweep

cudaError_t launch_bwd_close(int RP, const SweepBwdArgs &a, cudaStream_t st)
{
    using namespace sweep;
    return RP == 16 ? close_t<16>(a, st) : RP == 32 ? close_t<32>(a, st) : RP == 64 ? close_t<64>(a, st) : RP == 128 ? close_t<128>(a, st) : close_t<256>(a, st);
}

cudaError_t launch_bwd_assemble(int RP, const SweepBwdArgs &a, cudaStream_t st)
{
    using namespace sweep;
    return RP == 16 ? assemble_t<16>(a, st) : RP == 32 ? assemble_t<32>(a, st) : RP == 64 ? assemble_t<64>(a, st) : RP == 128 ? assemble_t<128>(a, st) : assemble_t<256>(a, st);
}

cudaError_t launch_bwd_reverse(const SweepPlan &P, const SweepBwdArgs &a, cudaStream_t st)
{
    using namespace sweep;
    switch (P.RP) {
    case 16: return reverse_t<16>(P, a, st);
    case 32: return reverse_t<32>(P, a, st);
    case 64: return reverse_t<64>(P, a, st);
    case 128: return reverse_t<128>(P, a, st);
    default: return reverse_t<256>(P, a, st);
    }
}

cudaError_t launch_bwd_merge(const float *part_q, const float *part_k, const float *dbeta_direct, const float *dbeta_acc, float *dz,
                             float *dbeta, int B, int H, int d, int r, int RP, int chunks, bool add, cudaStream_t st)
{
    const size_t threads = (size_t)H * r * d * 8;
    return chain_launch(sweep::merge_kernel, dim3((unsigned)((threads + 255) / 256)), 256, 0, st, part_q, part_k, dbeta_direct, dbeta_acc, dz, dbeta,
                        B, H, d, r, RP, chunks, add);
}

} // namespace lot
