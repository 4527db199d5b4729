// Sweep path: Sinkhorn iterations in scaling form on a float32 Gibbs kernel, all passes in one launch (lot_sweep.cu).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

namespace lot {

// Exponent range of the float32 Gibbs kernel.  A row's largest entry is 2^67 and a weight stays in [2^-110, 2^50]:
// products and row sums stay below 2^127, column sums nv beta / w in (2^-50, 2^127), and an entry that was flushed to
// zero (below 2^-126) is below 2^-24 of its row's sum whatever the weights (2^-126 2^50 256 against 2^67 2^-110).
// That is a window of 160 binades for the potentials before the kernel has to be rebuilt around them; the weights
// start in the middle of it.
constexpr float kKernelTop = 67.f, kStartLog2 = -50.f;

// Problem p of a sweep is side (p odd ? queries : keys) of slice p / 2, or with sides of different lengths, all of the longer one first;
// side 0 = queries, side 1 = keys.
struct SweepArgs {
    const void *x[2];        // [BH][n_side][d] tokens
    const float *z, *beta;   // [H][r][d], [H][r]
    const int32_t *key_len;  // [B] or nullptr (keys only)
    const float *mass[2];    // [BH][n_side] token weights or nullptr
    const float *g_in[2];    // [BH][r] starting potentials (natural units) or nullptr
    float *kt[2];            // [BH][n_side][RP] stabilised Gibbs kernel, columns >= r are zero
    float *inv[2];           // [BH][n_side] reciprocal row sums of the closing update (0: token without mass)
    float *w[2];             // [BH][RP] weights of the closing update: plan row i = kt[i][t] w[t] inv[i]
    double *gref[2];         // [BH][RP] reference potentials of kt, base-2 units
    float *g_out[2];         // [BH][r] potentials in natural units or nullptr
    unsigned long long *xbuf;   // exchange words of the groups (exchange_bytes; zero at the start of a call)
    float *hist;             // backward: [iters + 1][problems][RP] weights before every iteration and after the last, relative to
                             // the kernel as it is left, or nullptr
    double *hist_g;          // ... and the potentials themselves, of the problems whose kernel was rebuilt
    int *wide;               // ... [problems] 1: the kept weights leave float32's range, use hist_g
    uint4 *head;             // words that launch_build clears: status, tickets, exchange words
    size_t head_words;
    int *status;
    int B, H, d, r;
    int n[2];                // tokens per slice
    int skip;                // leading tokens of both sides that take no part (the class token)
    int C, K, groups;        // thread blocks per problem, per cluster (1: no clusters), problems in flight
    int srows;               // rows of a block's share that stay in shared memory
    int tcols;               // columns of tensor memory that take the next ones (0: none)
    int iters;
    int terms;               // bf16 tokens: terms a pivot is taken as in the first build (3: exact, 2)
    unsigned seq0;           // exchange sequence number this launch starts from
    double scale;            // log2(e)/eps
    double eps_ln2;
};

struct SweepPlan {
    int RP, C, K, groups, srows, tcols;
    int threads;             // of a block
    int chained;             // 1: may start behind its predecessor's last blocks
    size_t smem;
};

namespace sweep {
// the kernels of one type and use; a file each, compiled side by side
cudaError_t launch_f32(const SweepPlan &P, const SweepArgs &a, cudaStream_t st);
cudaError_t launch_bf16(const SweepPlan &P, const SweepArgs &a, cudaStream_t st);
cudaError_t launch_keep(const SweepPlan &P, const SweepArgs &a, cudaStream_t st);        // bf16, with the weights of every iteration
int cluster_count(int K, size_t smem);                                                   // clusters of K such blocks that run at once, 0: not known
}
int cluster_blocks(int K, int occ);      // blocks that run at once as clusters of K, `occ` to an SM
inline size_t exchange_bytes(int RP, int C, int K, int groups) { return C > K ? (size_t)groups * 2 * (C / K) * RP * 8 : 0; }
SweepPlan sweep_plan(int dtype, int BH, int nq, int nk, int d, int r, bool keep = false);      // keep: for the backward
constexpr int kWarpEntries = 4096;       // the most entries of a problem that one warp takes by itself
cudaError_t launch_build(int RP, const SweepArgs &a, int dtype, cudaStream_t st);
bool build_tc_supported(int RP, int d);  // bf16 tokens on tcgen05 (lot_build_tc.cu)
cudaError_t launch_build_tc(int RP, const SweepArgs &a, cudaStream_t st);
cudaError_t launch_sweep(const SweepPlan &P, const SweepArgs &a, int dtype, cudaStream_t st);

struct SweepApplyArgs {
    const float *kt[2], *inv[2], *w[2];   // inv, w: nullptr means 1 (kt is used as it is)
    const float *beta;       // nullptr: no scaling of W'
    const int32_t *key_len;
    const float *mass2;      // key weights or nullptr
    const void *v;
    void *out;
    float *wpart;            // [BH][chunks][r][d]
    float *Wp;               // [BH][r][d]; nullptr on the key side: the chunk partials are the result
    const int32_t *out_len;  // query side: rows beyond this length are zero, or nullptr
    unsigned *counter;
    int B, H, nq, nk, d, r, RP;
    int skip;                // leading tokens that take no part
    int terms;               // bf16 tensors: terms of a plan entry and of W' (3: float32 products, 2: hi + lo)
    int per_head;            // query side: Wp is [H][r][d]
    int chunks, rows_per_chunk;
};
// second: another product of the same sizes, buffers of its own, in the same launch (bf16 tensors)
cudaError_t launch_sweep_apply_w(const SweepApplyArgs &a, int dtype, cudaStream_t st, const SweepApplyArgs *second = nullptr);
cudaError_t launch_sweep_apply_out(const SweepApplyArgs &a, int dtype, cudaStream_t st);

// ---- backward of bf16 tensors on the stored kernel (lot_sweep_bwd.cu); problem numbering as above ----
struct SweepBwdArgs {
    SweepArgs s;             // x, z, kt, inv, w, hist, hist_g, wide, groups as in the forward; seq0 continues its sequence
    const void *g[2];        // [BH][n][d] bf16: dout (queries), v (keys)
    const float *wmat[2];    // [BH][r][d]: W' (queries), dW (keys): the plan's gradient is g . wmat
    float *dC[2];            // [BH][n][RP] gradient with respect to the similarities
    float2 *coef;            // [problems][T][n] row coefficients of every reverse step
    float *fk;               // [T][problems][RP] column coefficients
    float *gpart;            // [problems][tiles][RP] column sums of the closing step
    float *dbeta_acc;        // [problems][RP]
    int T, tiles;
    double eps;
};
// Everything behind the reverse steps: dx = dC Z, part = chunk partials of dC^T x (lot_sweep_grad.cu)
struct SweepGradArgs {
    SweepBwdArgs b;
    void *dx[2];             // [BH][n][d] bf16
    float *part[2];          // [BH][chunks][r][d]
    int chunks, rows;
};
bool sweep_grad_supported(int r, int d);
int sweep_grad_chunks(int BH, int n);                // of whole steps of 64 rows
cudaError_t launch_sweep_grad(int RP, const SweepGradArgs &a, cudaStream_t st);
cudaError_t launch_bwd_close(int RP, const SweepBwdArgs &a, cudaStream_t st);
cudaError_t launch_bwd_reverse(const SweepPlan &P, const SweepBwdArgs &a, cudaStream_t st);
cudaError_t launch_bwd_assemble(int RP, const SweepBwdArgs &a, cudaStream_t st);
// dz[h][t][c] = sum over batch, sides and chunks of the partials of dC^T x; dbeta as in launch_bwd_dz; add: on top of what they hold
cudaError_t launch_bwd_merge(const float *part_q, const float *part_k, const float *dbeta_direct, const float *dbeta_acc, float *dz,
                             float *dbeta, int B, int H, int d, int r, int RP, int chunks, bool add, cudaStream_t st);

} // namespace lot
