// Sweep path of the LOT attention (Eq. (1)-(2), scaling form): any supported shape, float32 or bf16 tensors, token
// weights, key lengths, starting potentials.
//
// A problem (one side of one slice) is shared by a group of C thread blocks.  lot_build.cu has left the stabilised Gibbs
// kernel K_it = 2^(L_it + Gref_t - ref_i) in global memory in float32; each block keeps the first `srows` rows of its
// share in shared memory (the rest stays in L2) and runs the iterations on them:
//   s_i = sum_t K_it w_t,   c_t = sum_i m_i K_it / s_i,   w_t <- target_t / c_t        (G_t = Gref_t + log2 w_t)
// two multiply-adds per entry and pass, no exponential and no logarithm.  Column sums are added lane -> warp -> block ->
// group in a fixed order; the blocks of a group exchange them through 64-bit words that carry a sequence number beside
// the value.  When a weight leaves its range (lot_sweep.h) the kernel is rebuilt around the current potentials; when a
// column sum itself leaves float32's range that iteration is redone in the log domain (column maxima first), so any
// spread of the potentials is exact.
// What bounds a pass: shared-memory reads (4 bytes per entry at 128 bytes per clock and SM) and, for C > 1, one or two
// round trips through L2 for the exchange, which other blocks on the SM (other groups) hide.
#include "lot_chain.cuh"
#include "lot_sweep_core.cuh"

#include <mutex>

namespace lot {
namespace sweep {

// Closing update and results of problem p.  Out of line, and everything worked out again: nothing of the problem is live
// across recover() and this call, which would cost the iteration loop its registers (spills in it: a fifth slower).
template <typename T, int RP, int CPL, int THREADS>
__device__ __noinline__ void finish(const SweepArgs *ap, int p, int c)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const SweepArgs &a = *ap;
    const Shared S = carve<T, RP, THREADS>(smem, a.srows);
    Share R;
    const Problem P = locate<RP, CPL, THREADS>(a, p, c, R);
    const int tid = threadIdx.x;
    if (a.close && P.nv > 0) {
        const Lane<RP, CPL> L = make_lane<RP, CPL>(S);
        u64 w[CPL / 2], acc[CPL / 2];
        load_weights<RP, CPL>(L, w);
        pass<RP, CPL, THREADS, true>(L, R, w, acc, a.inv[P.side] + (size_t)P.slice * P.n + P.row0);
    }
    if (c == 0 && tid < RP) {
        const double gl = S.gref[tid];
        const float wl = tid < a.r ? S.w[tid] : 0.f;
        a.w[P.side][(size_t)P.slice * RP + tid] = wl;
        a.gref[P.side][(size_t)P.slice * RP + tid] = gl;
        if (a.close && tid < a.r && a.g_out[P.side] != nullptr)
            a.g_out[P.side][(size_t)P.slice * a.r + tid] = (float)((gl + log2((double)wl)) * a.eps_ln2);
    }
}

// KEEP: the weights of every iteration go to a.hist (backward).
template <typename T, int RP, int CPL, int THREADS, bool GROUP, bool KEEP>
__global__ void __launch_bounds__(THREADS, max_blocks(CPL, THREADS))
sweep_kernel(const __grid_constant__ SweepArgs a)
{
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x, group = GROUP ? blockIdx.x / a.C : blockIdx.x, c = GROUP ? blockIdx.x % a.C : 0;
    const int NP = 2 * a.B * a.H, r = a.r;
    unsigned seq = a.seq0;
    const Shared S = carve<T, RP, THREADS>(smem, a.srows);
    if (tid == 0) { S.flag[0] = 0; S.flag[1] = 0; }
    chain_wait();

    for (int p = group; p < NP; p += a.groups) {
        Share R;
        const Problem P = locate<RP, CPL, THREADS>(a, p, c, R);
        __syncthreads();                                     // the previous problem is done with shared memory
        if (tid < RP) {
            double g0 = -(double)kStartLog2;
            float w0 = tid < r ? kStart : 0.f;
            if (!a.first) {
                g0 = a.gref[P.side][(size_t)P.slice * RP + tid];
                w0 = a.w[P.side][(size_t)P.slice * RP + tid];
            } else if (tid < r && a.g_in[P.side] != nullptr) {
                g0 += (double)__ldg(a.g_in[P.side] + (size_t)P.slice * r + tid) * a.scale;
            }
            S.gref[tid] = g0;
            S.w[tid] = w0;
            S.tgt[tid] = tid < r ? __ldg(a.beta + P.h * r + tid) * (R.mass ? 1.f : (float)P.nv) : 0.f;
        }
        load_rows<RP, CPL, THREADS>(S, R);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (P.nv <= 0 && tid == 0 && a.first && c == 0) atomicOr(a.status, 2 /* LOT_DEV_EMPTY */);
        __syncthreads();
        float wold = 0.f, wnew = S.w[tid < RP ? tid : 0];
        bool bad = false;
        int it = a.it0;
        if (P.nv > 0) {
            const Lane<RP, CPL> L = make_lane<RP, CPL>(S);
            const float tgt = S.tgt[tid < RP ? tid : 0];
            u64 w[CPL / 2];
            load_weights<RP, CPL>(L, w);
            float *hp = KEEP && c == 0 && tid < RP ? a.hist + (size_t)p * RP + tid : nullptr;      // thread t's column
            if (KEEP && hp != nullptr) *hp = S.w[tid];
            for (; it < a.it1; ++it) {
                bad = iterate<RP, CPL, THREADS, GROUP>(a, S, R, L, w, tgt, group, c, seq, wold, wnew);
                if (bad) break;
                if (KEEP && hp != nullptr) {
                    hp += (size_t)NP * RP;
                    *hp = tid < r ? wnew : 0.f;
                }
            }
            if (KEEP && !bad && c == 0 && tid == 0) a.wide[p] = 0;
        }
        if (bad) seq = recover<T, RP, CPL, THREADS, GROUP>(&a, p, group, c, it, seq, wold, wnew);
        if (p + a.groups >= NP) chain_next();
        finish<T, RP, CPL, THREADS>(&a, p, c);
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------------------------
constexpr int kSmPerBlockReserve = 1024, kSmemPerSM = 228 * 1024, kSmemPerBlock = 227 * 1024;

template <typename T, int RP, int CPL, int THREADS, bool GROUP, bool KEEP>
static cudaError_t launch_g(const SweepPlan &P, const SweepArgs &a, cudaStream_t st)
{
    auto kern = sweep_kernel<T, RP, CPL, THREADS, GROUP, KEEP>;
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
    if (!GROUP) {
        return chain_launch(kern, grid, THREADS, P.smem, st, a);
    }
    SweepArgs copy = a;
    void *args[] = {&copy};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(kern), grid, dim3(THREADS), args, P.smem, st);
}

template <typename T, int RP>
static cudaError_t launch_t(const SweepPlan &P, const SweepArgs &a, cudaStream_t st)
{
    if constexpr (sizeof(T) == 2) {                          // the backward of float32 tensors keeps its own history
        if (a.hist != nullptr)
            return P.C > 1 ? launch_g<T, RP, wide_cols(RP), 256, true, true>(P, a, st) : launch_g<T, RP, wide_cols(RP), 256, false, true>(P, a, st);
    }
    return P.C > 1 ? launch_g<T, RP, wide_cols(RP), 256, true, false>(P, a, st) : launch_g<T, RP, wide_cols(RP), 256, false, false>(P, a, st);
}

template <typename T>
static cudaError_t launch_rp(const SweepPlan &P, const SweepArgs &a, cudaStream_t st)
{
    switch (P.RP) {
    case 16: return launch_t<T, 16>(P, a, st);
    case 32: return launch_t<T, 32>(P, a, st);
    case 64: return launch_t<T, 64>(P, a, st);
    case 128: return launch_t<T, 128>(P, a, st);
    default: return launch_t<T, 256>(P, a, st);
    }
}

} // namespace sweep

cudaError_t launch_sweep(const SweepPlan &P, const SweepArgs &a, int dtype, cudaStream_t st)
{
    return dtype == 0 ? sweep::launch_rp<float>(P, a, st) : sweep::launch_rp<__nv_bfloat16>(P, a, st);
}

// Blocks per problem and where the rows live: the split with the least modelled time.  A round (all resident groups
// finish one problem each) costs its build plus, per iteration, the larger of one block's latency chain and the SM's
// shared-memory and issue time; see the comment at the constants for what they come from.
SweepPlan sweep_plan(int dtype, int BH, int nq, int nk, int d, int r)
{
    using namespace sweep;
    const int P = 2 * BH, n = nq > nk ? nq : nk, sms = device_sm_count();
    // a program asks for the same sizes again and again (workspace query, then the call): the last answer is kept
    struct Memo { int key[7]; SweepPlan plan; };
    static thread_local Memo memo = {};
    const int key[7] = {dtype + 1, BH, nq, nk, d, r, sms};
    if (memcmp(key, memo.key, sizeof(key)) == 0) return memo.plan;
    SweepPlan best{};
    best.RP = r <= 16 ? 16 : r <= 32 ? 32 : r <= 64 ? 64 : r <= 128 ? 128 : 256;
    const int RP = best.RP, CPL = wide_cols(RP), threads = 256;
    double best_t = 1e30;
    for (int occ = 1; occ <= max_blocks(CPL, threads); ++occ) {
        const int step = threads * CPL / RP;                                  // rows per step of a block
        const size_t f0 = fixed_bytes<float>(RP, threads), f1 = fixed_bytes<__nv_bfloat16>(RP, threads), fixed = f0 > f1 ? f0 : f1;
        size_t per_block = (size_t)kSmemPerSM / occ - kSmPerBlockReserve;
        if (per_block > (size_t)kSmemPerBlock) per_block = kSmemPerBlock;
        const int cap = (int)((per_block - fixed) / ((size_t)RP * 4)) / step * step;
        const int all_slots = sms * occ;
        // every group size up to 32 blocks, then those that divide the blocks into whole groups
        for (int C = 1; C <= all_slots && C <= (n + 15) / 16; C = C < 32 ? C + 1 : all_slots / C > 1 ? all_slots / (all_slots / C - 1) : all_slots + 1) {
            const int rows = (n + C - 1) / C, up = (rows + step - 1) / step * step, srows = up < cap ? up : cap;
            const size_t smem = fixed + (size_t)srows * RP * 4;
            int fit = (int)((size_t)kSmemPerSM / (smem + kSmPerBlockReserve));
            if (fit > occ) fit = occ;
            const int slots = sms * (C == 1 ? fit : occ);
            int groups = C == 1 ? P : slots / C;
            if (groups > P) groups = P;
            const int resident = C == 1 ? (P < slots ? P : slots) : groups * C;
            const int rounds = C == 1 ? (P + slots - 1) / slots : (P + groups - 1) / groups;
            const double per_sm = (double)((resident + sms - 1) / sms);       // blocks that share an SM
            // us: SM time per entry (issue and shared-memory reads), twice that for a block alone on its SM; the latency of an
            // iteration with its exchange; streamed rows at the L2's rate, at the HBM's when all of them exceed the L2, and
            // never faster than one SM reads.  The constants are fitted to the times of whole calls, the last two lines of
            // latency and the rate of one SM to those of 64 problems of 16384 rows at RP = 256 over C (sweep kernel, 20
            // iterations: 4152 us at 42, 3833 at 49, 3957 at 59, 4312 at 74, 4877 at 98, 5947 at 148).  Measured by itself
            // (group_columns) the latency is 4.9 at 49 blocks, 5.6 at 74, 7.7 at 148 with owners, where the line says 5.2,
            // 5.6, 7.0; without them the line is too low from 8 blocks on (16 blocks at RP = 256: 3.7, line 2.5).
            const double entry = (RP <= 32 ? 0.055 : 0.045) / 1900.0;
            const double lat = C == 1 ? 0.45 : C * RP <= kDirectWords ? 0.9 + 0.4 * C * RP / 1024.0 : 4.3 + 0.018 * C;
            const double mine = 2.0 * rows * RP * entry, sm_us = per_sm * rows * RP * entry;
            const double glob = (double)(rows > srows ? rows - srows : 0) * RP * 4.0, all = glob * resident;
            double it = lat + mine;
            if (sm_us > it) it = sm_us;
            const double gl_us = all / (all > 90e6 ? 5.5e6 : 10e6), gl_sm = per_sm * glob / 70e3;
            it += gl_us > gl_sm ? gl_us : gl_sm;
            const double t = rounds * (12 * it + 3.0);
            if (t < best_t) {
                best_t = t;
                best.C = C; best.groups = groups; best.srows = srows;
                best.smem = smem;
            }
        }
    }
    best.steps = 0;
    if (dtype == 0 && (double)P / 2 * ((double)nq + nk) * RP * 4.0 > 2.0 * sms * kSmemPerBlock) {
        // float32 kernel far larger than shared memory: every pass streams it, one launch per pass
        const int slots = 2 * sms;
        best.C = slots / P < 1 ? 1 : slots / P;
        if (best.C > (n + 15) / 16) best.C = (n + 15) / 16;
        best.groups = best.C == 1 ? P : (slots / best.C < P ? slots / best.C : P);
        best.srows = 0;
        best.smem = fixed_bytes<__nv_bfloat16>(RP, 256);
        best.steps = 1;
    }
    memcpy(memo.key, key, sizeof(key));
    memo.plan = best;
    return best;
}

} // namespace lot
