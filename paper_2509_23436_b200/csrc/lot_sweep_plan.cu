// Host side of the sweep path (lot_sweep.cu): how a call's problems are split over the device.
#include "lot_sweep_core.cuh"

#include <mutex>

namespace lot {
namespace sweep {

// Shared memory a block may take with `occ` of them to an SM.
static size_t block_smem(int occ)
{
    const size_t s = (size_t)kSmemPerSM / occ - kSmPerBlockReserve;
    return s < (size_t)kSmemPerBlock ? s : (size_t)kSmemPerBlock;
}

} // namespace sweep

cudaError_t launch_sweep(const SweepPlan &P, const SweepArgs &a, int dtype, cudaStream_t st)
{
    // the backward of float32 tensors keeps its own history
    return dtype == 0 ? sweep::launch_f32(P, a, st) : a.hist != nullptr ? sweep::launch_keep(P, a, st) : sweep::launch_bf16(P, a, st);
}

// Blocks that run at once as clusters of K with `occ` to an SM: a cluster's blocks share a GPC, so some slots stay empty (of 148 SMs
// with one block each 148, 132 and 120 work in clusters of 2, 4 and 8, with two 296, 284 and 264).  Asked for once per device;
// a host without one gets an estimate.
int cluster_blocks(int K, int occ)
{
    using namespace sweep;
    static std::mutex mu;
    static int known[64][kPeers + 1][4] = {};
    const int estimate = device_sm_count() * occ * 7 / 8 / K * K;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return estimate; }
    std::lock_guard<std::mutex> lock(mu);
    int &blocks = known[dev][K][occ];
    if (blocks == 0) blocks = cluster_count(K, block_smem(occ)) * K;
    return blocks > 0 ? blocks : estimate;
}

// Blocks per problem and where the rows live: the split with the least modelled time.  In a round all resident groups finish
// one problem each; it costs the reading of its rows and, per iteration, the larger of one block's chain (latency with
// the exchange, its own steps) and of what the blocks of an SM need together.  The constants are fitted to the times of whole calls of 12
// iterations: 108 sizes from 2 problems of 300 tokens to 512 of 1100 and 18 of 52000, each in up to 56 forced splits; over those, the
// split chosen is on average 1.0 % slower than the best one, and in 8 of them more than 5 % (22 % at most: 32 problems of 700 tokens, where
// clusters of four take 13 us longer than of three for no reason this model knows).
// Rows in tensor memory are what it mostly takes where a problem is more than one block's shared memory: a pass over rows there
// runs at 26 entries a clock and SM against 18 from shared memory alone (a loop of passes at RP = 256), and 480 KB instead of 227
// stay on an SM.  Where all rows fit shared memory, 512 threads are worth it at RP <= 32 with a block a problem (64 slices of 700 at r = 32
// 47.4 us, 256 threads 49.3) and not for clusters (8 of 500 at r = 64, T = 20: 55.6, 49.6).
namespace sweep {
// Whether groups of one cluster may start behind the predecessor's last blocks, which saves 2 to 4 us of a call.  Placed while those
// hold parts of the SMs, clusters leave gaps, and where nearly all of a device's are asked for the last ones wait for the first to
// end: float32, r = 64, 90 rows a block, us an iteration, chained / ordinary: 82 clusters of three of 93 that fit two to an SM 2.37 / 1.09, 32
// of 33 of eight 2.36 / 0.90; one block to an SM, 44 of 45 of three 1.91 / 1.21, 26 of 26 of five 2.40 / 1.16, but of two, four
// and eight the same up to the last; three to an SM (r = 16) 142 of 142 of three 2.09 / 1.15, 66 of 71 of six 1.41 / 1.17, 44 of 48 of
// eight 1.17 / 1.19, 126 of 142 of three 1.13 / 1.20 (cross-attention 333 x 1531 at r = 32, 128 of 142: 76.4 / 79.7 a call).  Two to an
// SM they also lie unevenly well below that (12 slices of 2500 at r = 64, T = 20: 118.6 / 114.5).
constexpr bool chain_fits(int groups, int K, int occ, int slots)
{
    return occ == 1 ? K % 2 == 0 || 5 * groups * K <= 4 * slots : occ == 3 && 12 * groups * K <= 11 * slots;
}
constexpr double kIters = 12, kClockMHz = 1900;
constexpr double kEntryClk[2][2] = {{0.032, 0.037}, {0.046, 0.041}};      // clocks of an SM per entry: [512 threads][RP <= 32]
constexpr double kAloneBlock = 1.7;      // times as many where a block of 256 threads has the SM to itself
constexpr double kOrdinaryStart = 2.9;   // us
// What a block's rows may cost to rebuild, us per row, column and channel with 256 threads, weighed by how seldom calls do: the fit's calls never
// did, and without it peaked ones were given few blocks of many rows (39 slices of 3059 at r = 32, eps 0.02 205 us before that fit, 323 with it;
// 12 of 1047 at d = 128, r = 16 64 and 80).  Over 774 drawn calls, a quarter of them peaked, against the splits before: peaked 2.6 % faster
// on average with it and 1.4 without, others 3.1 and 3.1; 30 in all instead of 48 more than 2 % slower.  A third and one and a half
// times of it are no better.
constexpr double kRebuild = 3e-6;
}

SweepPlan sweep_plan(int dtype, int BH, int nq, int nk, int d, int r, bool keep)
{
    using namespace sweep;
    const int P = 2 * BH, n = nq > nk ? nq : nk, sms = device_sm_count();
    // a program asks for the same sizes again and again (workspace query, then the call; its layers in turn): the last answers are kept
    struct Memo { int key[8]; SweepPlan plan; };
    static thread_local Memo memos[8] = {};
    static thread_local unsigned next = 0;
    const int key[8] = {dtype + 1, BH, nq, nk, d, r, sms, keep};
    for (const Memo &m : memos)
        if (memcmp(key, m.key, sizeof(key)) == 0) return m.plan;
    SweepPlan best{};
    best.RP = r <= 16 ? 16 : r <= 32 ? 32 : r <= 64 ? 64 : r <= 128 ? 128 : 256;
    const int RP = best.RP;
    double best_t = 1e30;
    auto consider = [&](bool tensor, int occ, int C, int K, int slots) {
        const int threads = tensor ? kTensorThreads : 256, CPL = tensor ? kTensorLane : wide_cols(RP);
        const double entry = kEntryClk[tensor][RP <= 32] / kClockMHz * (tensor ? 1.0 : kAloneBlock);
        double lat = tensor ? (C == 1 ? 0.88 : 0.98) + RP * (1.2 / 256) : 0.79 + RP * (0.87 / 256);
        if (C > 1) {
            lat += C == K ? 0.67 + 0.025 * (K - 2) : 2.2 + 0.33 * (occ - 1);
            // most splits are no match for the best so far by this alone (a search of all of them took 60 us)
            if (slots < C) return;
            const int fly = slots / C < P ? slots / C : P, turns = ((nq == nk ? P : BH) + fly - 1) / fly;
            if (turns * (kIters + 0.7) * (lat + (double)n / C * RP * entry) >= best_t) return;
        }
        const int step = threads * CPL / RP;                                  // rows per step of a block
        const size_t f0 = fixed_bytes<float>(RP, threads), f1 = fixed_bytes<__nv_bfloat16>(RP, threads);
        const size_t fixed = (f0 > f1 ? f0 : f1) + (size_t)peer_bytes(RP, C, K);
        const int cap = (int)((block_smem(occ) - fixed) / ((size_t)RP * 4)) / step * step;
        const int rows = (n + C - 1) / C, up = (rows + step - 1) / step * step, srows = up < cap ? up : cap;
        size_t smem = fixed + (size_t)srows * RP * 4;
        int fit = (int)((size_t)kSmemPerSM / (smem + kSmPerBlockReserve));
        if (fit > occ) fit = occ;
        if (C == 1) slots = sms * fit;
        int groups = C == 1 ? P : slots / C;
        if (groups > P) groups = P;
        if (groups < 1) return;
        const int fly = C == 1 && P > slots ? slots : groups, resident = fly * C;            // problems and blocks at once
        const int per_sm = (resident + sms - 1) / sms;                        // blocks that share an SM
        // blocks that could have an SM each do: a chained start would put some of them two to an SM
        const int single = C == 1 ? sms : cluster_blocks(K, 1);
        if (resident <= single && smem < kAloneSmem) smem = kAloneSmem;
        const bool chained = C == 1 || (C == K && (resident <= single ? chain_fits(groups, K, 1, single) : chain_fits(groups, K, occ, slots)));
        const int tcols = tensor && rows > srows ? kTensorCols : 0, trows = tcols / (threads / 128) / CPL * step;
        // Rows of 16 columns: no more than a few per cent of them streamed beside tensor memory.  The model takes such splits for the better ones, and a
        // block of that many rows is slow to rebuild them: 32 slices of 16384 tokens at d = 128, r = 16, two blocks of 8192 rows a problem 390 us,
        // peaked 578, four of 4096 384 and 485 (before tensor memory 451 and 498).
        if (tensor && RP == 16 && rows > 1.05 * (srows + trows)) return;
        // us of a problem of m tokens
        auto problem = [&](int m) {
            const int mine = (m + C - 1) / C, ns = mine < srows ? mine : srows, nt = mine - ns < trows ? mine - ns : trows, rest = mine - ns - nt;
            const int steps = (ns + step - 1) / step + (nt + 2 * step - 1) / (2 * step) * 2 + (rest + 2 * step - 1) / (2 * step) * 2;
            const double work = (double)steps * step * RP * kEntryClk[tensor][RP <= 32] / kClockMHz;
            double it = lat + work * (tensor ? 1.0 : kAloneBlock);
            if (it < per_sm * work) it = per_sm * work;
            if (rest > 0) {
                const double mb = rest * (RP * 4e-6), all = mb * resident;
                const double l2 = all / (all > 60 ? 5.0 : 11.0), sm = per_sm * mb / 0.08;       // TB/s: L2 beyond half of it is no faster than memory
                it += 0.9 + (l2 > sm ? l2 : sm);
            }
            return (kIters + 0.7) * it + resident * (double)(ns + nt) * (RP * 4e-6) / 7.5 + mine * (RP * 8e-5) + (double)mine * RP * d * (kRebuild * 256 / threads) + 3.0;
        };
        const int rounds = (P + fly - 1) / fly, first = nq == nk ? rounds : (BH + fly - 1) / fly;         // the longer side's come first
        const double t = first * problem(n) + (rounds > first ? (rounds - first) * problem(nq < nk ? nq : nk) : 0.0) + (chained ? 0.0 : kOrdinaryStart) +
                         (tensor ? 0.9 : 0.0);
        if (t < best_t) {
            best_t = t;
            best.C = C; best.K = K; best.groups = groups; best.srows = srows;
            best.smem = smem; best.tcols = tcols; best.threads = threads;
            best.chained = chained;
        }
    };
    // More short problems than blocks of 256 threads fit at once: one warp each, whose barriers wait for nobody and whose sums end in the
    // warp.  float32, d = 64, T = 20, us, blocks / warps: 384 slices of 64 tokens at r = 16 51.8 / 35.3, of 128 60.0 / 49.0, of 256 88.8 / 82.3,
    // 512 of 128 at r = 32 109 / 93; but 384 of 500 at r = 16 147 / 152, and 3 of 128 at r = 16 27.2 / 33.3.
    const bool warp = !keep && RP <= 32 && (long long)n * RP <= kWarpEntries && P > 3 * sms;
    for (int form = 0; !warp && form <= max_blocks(wide_cols(RP), 256); ++form) {      // 0: with tensor memory, one block to an SM
        const bool tensor = form == 0;
        const int occ = tensor ? 1 : form, threads = tensor ? kTensorThreads : 256, half = threads * (tensor ? kTensorLane : wide_cols(RP)) / RP / 2;
        const int most = (n + half - 1) / half;                               // half a step's rows a block at least
        consider(tensor, occ, 1, 1, 0);
        for (int K = 2; K <= kPeers; ++K) {
            const int slots = cluster_blocks(K, occ), all = slots / K;
            if (K <= most) consider(tensor, occ, K, K, slots);
            if ((K & (K - 1)) == 0)                                           // several clusters
                for (int M = 2; M <= all && M <= kWords && M * K <= most; ++M) consider(tensor, occ, M * K, K, slots);
        }
    }
    if (warp) {
        const int step = 32 * wide_cols(RP) / RP;
        const size_t f0 = fixed_bytes<float>(RP, 32), f1 = fixed_bytes<__nv_bfloat16>(RP, 32);
        best.C = best.K = 1; best.groups = P; best.srows = (n + step - 1) / step * step; best.tcols = 0; best.threads = 32; best.chained = 1;
        best.smem = (f0 > f1 ? f0 : f1) + (size_t)best.srows * RP * 4;
    }
    Memo &m = memos[next++ % 8];
    memcpy(m.key, key, sizeof(key));
    m.plan = best;
    return best;
}

} // namespace lot
