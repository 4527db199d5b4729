// Sweep path: Sinkhorn iterations in scaling form on a float32 Gibbs kernel, several passes per launch (lot_sweep.cu).
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
constexpr int kSweepCopies = 8;     // places the totals of an exchange are left in

// Problem p of a sweep is side (p odd ? queries : keys) of slice p / 2; side 0 = queries, side 1 = keys.
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
    unsigned long long *xbuf;   // exchange words of the groups (zero at the start of the first launch of a call)
    unsigned long long *ybuf;
    int *status;
    int B, H, d, r;
    int n[2];                // tokens per slice
    int skip;                // leading tokens of both sides that take no part (the class token)
    int C, groups;           // thread blocks per problem, problems in flight
    int srows;               // rows of a block's share that stay in shared memory
    int it0, it1;            // iterations this launch runs
    int first, close;        // start from the given potentials (else from the state in w, gref) / closing update last
    unsigned seq0;           // exchange sequence number this launch starts from
    double scale;            // log2(e)/eps
    double eps_ln2;
};

struct SweepPlan {
    int RP, C, groups, srows;
    int steps;               // 1: one launch per iteration (the kernel streams from global memory anyway)
    size_t smem;
};

SweepPlan sweep_plan(int dtype, int BH, int nq, int nk, int d, int r);
cudaError_t launch_build(int RP, const SweepArgs &a, int dtype, int sides, cudaStream_t st);
cudaError_t launch_sweep(const SweepPlan &P, const SweepArgs &a, int dtype, cudaStream_t st);

struct SweepApplyArgs {
    const float *kt[2], *inv[2], *w[2];
    const float *beta;
    const int32_t *key_len;
    const float *mass2;      // key weights or nullptr
    const void *v;
    void *out;
    float *wpart;            // [BH][chunks][r][d]
    float *Wp;               // [BH][r][d]
    unsigned *counter;
    int B, H, nq, nk, d, r, RP;
    int skip;                // leading tokens that take no part
    int chunks, rows_per_chunk;
};
cudaError_t launch_sweep_apply_w(const SweepApplyArgs &a, int dtype, cudaStream_t st);
cudaError_t launch_sweep_apply_out(const SweepApplyArgs &a, int dtype, cudaStream_t st);

} // namespace lot
