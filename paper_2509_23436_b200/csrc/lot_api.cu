// The C ABI of liblot (see include/lot.h): argument validation, workspace carving and the
// launch sequence.  No arithmetic of the method lives here.
#include "../../include/lot.h"
#include "lot_internal.h"
#include "lot_sweep.h"

#include <math.h>
#include <atomic>
#include <mutex>
#include <unordered_map>

namespace {

using namespace lot;

constexpr int kMaxR = 256;
constexpr int kMaxD = 256;
constexpr int kMaxDevices = 64;

inline size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }
inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_dims(int B, int H, int n, int r)
{
    if (B < 0 || H < 1 || n < 0 || r < 1) return LOT_ERR_INVALID_ARG;
    if (r > kMaxR) return LOT_ERR_UNSUPPORTED_SHAPE;
    if ((long long)B * H > 32767) return LOT_ERR_UNSUPPORTED_SHAPE;
    if ((long long)n * r >= (1ll << 31)) return LOT_ERR_UNSUPPORTED_SHAPE;
    return LOT_OK;
}

int check_d(int n, int d)
{
    if (d < 1) return LOT_ERR_INVALID_ARG;
    if (d < 8 || d > kMaxD || (d % 8) != 0) return LOT_ERR_UNSUPPORTED_SHAPE;
    if ((long long)n * d >= (1ll << 31)) return LOT_ERR_UNSUPPORTED_SHAPE;
    return LOT_OK;
}

// Workspace of one Sinkhorn problem set.  The head (status word, potentials, tickets) is one
// contiguous region cleared at the start of every call.
struct SinkLayout {
    size_t status, G, counter, head_end, gnat, part, M, total;
    int chunks, rows_per_chunk;
};

// lt = bytes of the type potentials and row log-sum-exps are held in (4 or 8).
SinkLayout sink_layout(int nprob, int n, int r, size_t base, size_t lt)
{
    SinkLayout L;
    L.chunks = pass_chunks(nprob > 0 ? nprob : 1, n > 0 ? n : 1);
    L.rows_per_chunk = (n + L.chunks - 1) / L.chunks;
    size_t o = base;
    L.status = o; o += 256;
    L.G = o; o += up256((size_t)nprob * r * lt);
    L.counter = o; o += up256((size_t)nprob * 4);
    L.head_end = o;
    L.gnat = o; o += up256((size_t)nprob * r * 4);
    L.part = o; o += up256((size_t)nprob * L.chunks * r * 2 * 4);
    L.M = o; o += up256((size_t)nprob * n * lt);
    L.total = o;
    return L;
}

// Workspace of a forward on the general path (queries and keys may differ in number): the head (status word, tickets of
// the apply stage, exchange words of the sweep) is one region cleared at the start of every call.
struct ForwardLayout {
    SweepPlan plan;
    size_t counter, xbuf, head_end, w[2], gref[2], inv[2], kt[2], scores, wpart, Wp, total;
    int achunks, arows;
};

ForwardLayout forward_layout(int B, int H, int nq, int nk, int d, int r, int dtype, bool variant)
{
    ForwardLayout L;
    const int BH = B * H, n[2] = {nq, nk};
    L.plan = sweep_plan(dtype, BH > 0 ? BH : 1, nq > 0 ? nq : 1, nk > 0 ? nk : 1, d, r);
    const int RP = L.plan.RP;
    size_t o = 256;                                                   // status word at 0
    L.counter = o; o += up256((size_t)((r + 63) / 64) * ((d + 63) / 64) * BH * 4);
    L.xbuf = o;
    o += up256(exchange_bytes(RP, L.plan.C, L.plan.K, L.plan.groups));
    L.head_end = o;
    for (int side = 0; side < 2; ++side) {
        L.w[side] = o; o += up256((size_t)BH * RP * 4);
        L.gref[side] = o; o += up256((size_t)BH * RP * 8);
        L.inv[side] = o; o += up256((size_t)BH * n[side] * 4);
        L.kt[side] = o; o += up256((size_t)BH * n[side] * RP * 4);
    }
    L.scores = o;
    if (variant) o += up256((size_t)BH * nk * 4);
    L.achunks = apply_chunks(BH > 0 ? BH : 1, nk > 0 ? nk : 1, r, dtype == LOT_F32 ? d : 64);   // bf16: all channels in a block
    L.arows = (nk + L.achunks - 1) / L.achunks;
    L.wpart = o; o += up256((size_t)BH * L.achunks * r * d * 4);
    L.Wp = o; o += up256((size_t)BH * r * d * 4);
    // float32 tensors: never less than eight bytes per similarity, the size the interface has always asked for there
    const size_t least = dtype == LOT_F32 ? up256((size_t)BH * ((size_t)nq + nk) * r * 8) : 0;
    L.total = o > least ? o : least;
    return L;
}

// Workspace of lot_attention_bwd for float32 tensors: similarities in float64, the blocks of the log-domain passes, the
// kept potentials of every iteration, the gradient with respect to the similarities and the small reduction buffers.
struct BwdLayout {
    size_t counter, counter2, hist, gamma, dbeta_acc, head_end, part, M, cost, dC, wpart, Wp, Xw, dWm, dbeta_direct, zt,
        dzpart, total;
    int chunks, rows_per_chunk, achunks, arows, dzchunks;
};

BwdLayout bwd_layout(int B, int H, int n, int d, int r, int iters)
{
    BwdLayout L;
    const size_t lt = 8;
    const int BH = B * H, np = 2 * BH;
    const int tiles = ((r + 63) / 64) * ((d + 63) / 64) * BH;
    L.chunks = pass_chunks(np > 0 ? np : 1, n > 0 ? n : 1);
    L.rows_per_chunk = (n + L.chunks - 1) / L.chunks;
    L.achunks = apply_chunks(BH > 0 ? BH : 1, n > 0 ? n : 1, r, d);
    L.arows = (n + L.achunks - 1) / L.achunks;
    L.dzchunks = bwd_dz_chunks(BH > 0 ? BH : 1, n > 0 ? n : 1, r, d);
    size_t o = 256;                                   // status word at 0
    L.counter = o; o += up256((size_t)np * 4);
    L.counter2 = o; o += up256((size_t)tiles * 4);
    L.hist = o; o += up256((size_t)(iters + 1) * np * r * lt);
    L.gamma = o; o += up256((size_t)np * r * lt);
    L.dbeta_acc = o; o += up256((size_t)np * r * lt);
    L.head_end = o;
    L.part = o; o += up256((size_t)np * L.chunks * r * 8);
    L.M = o; o += up256((size_t)np * n * lt);
    L.cost = o; o += up256((size_t)np * n * r * lt);
    L.dC = o; o += up256((size_t)np * n * r * lt);
    L.wpart = o; o += up256((size_t)BH * L.achunks * r * d * 4);
    L.Wp = o; o += up256((size_t)BH * r * d * 4);
    L.Xw = o; o += up256((size_t)BH * r * d * 4);
    L.dWm = o; o += up256((size_t)BH * r * d * 4);
    L.dbeta_direct = o; o += up256((size_t)BH * r * 4);
    L.zt = o; o += up256((size_t)H * r * d * 4);
    L.dzpart = o; o += up256((size_t)np * L.dzchunks * r * d * lt);
    L.total = o;
    return L;
}

// Workspace of lot_attention_bwd for bf16 tensors: the forward's blocks (kernel and weights of both sides), the kept
// weights of every iteration, the row and column coefficients of the reverse steps and the gradient with respect to the
// similarities.
struct BwdSweepLayout {
    SweepPlan plan;
    int rounds, tiles, achunks, arows, gchunks, grows;
    size_t counter, xbuf, head_end, w[2], gref[2], inv[2], kt[2], dC[2], hist, hist_g, wide, coef, fk, gpart, dbeta_acc, wpart,
        wpart2, counter2, Wp, Xw, dWm, dbeta_direct, zpart[2], total;
};

BwdSweepLayout bwd_sweep_layout(int B, int H, int n, int d, int r, int iters)
{
    BwdSweepLayout L;
    const int BH = B * H > 0 ? B * H : 1, NP = 2 * BH;
    if (n < 1) n = 1;
    L.plan = sweep_plan(LOT_BF16, BH, n, n, d, r, true);
    const int RP = L.plan.RP;
    L.rounds = (NP + L.plan.groups - 1) / L.plan.groups;
    L.tiles = (n + 127) / 128;
    size_t o = 256;                                                   // status word at 0
    L.counter = o; o += up256((size_t)((r + 63) / 64) * ((d + 63) / 64) * BH * 4);
    L.counter2 = o; o += up256((size_t)((r + 63) / 64) * ((d + 63) / 64) * BH * 4);
    L.xbuf = o;
    o += up256(exchange_bytes(RP, L.plan.C, L.plan.K, L.plan.groups));
    L.head_end = o;
    for (int side = 0; side < 2; ++side) {
        L.w[side] = o; o += up256((size_t)BH * RP * 4);
        L.gref[side] = o; o += up256((size_t)BH * RP * 8);
        L.inv[side] = o; o += up256((size_t)BH * n * 4);
        L.kt[side] = o; o += up256((size_t)BH * n * RP * 4);
        L.dC[side] = o; o += up256((size_t)BH * n * RP * 4);
    }
    L.hist = o; o += up256((size_t)(iters + 1) * NP * RP * 4);
    L.hist_g = o; o += up256((size_t)(iters + 1) * NP * RP * 8);
    L.wide = o; o += up256((size_t)NP * 4);
    L.coef = o; o += up256((size_t)NP * iters * n * 8);
    L.fk = o; o += up256((size_t)iters * NP * RP * 4);
    L.gpart = o; o += up256((size_t)NP * L.tiles * RP * 4);
    L.dbeta_acc = o; o += up256((size_t)NP * RP * 4);
    L.achunks = apply_chunks(BH, n, r, 64);
    L.arows = (n + L.achunks - 1) / L.achunks;
    L.gchunks = sweep_grad_chunks(BH, n);
    L.grows = ((n + 63) / 64 + L.gchunks - 1) / L.gchunks * 64;
    L.wpart = o; o += up256((size_t)BH * L.achunks * r * d * 4);
    L.wpart2 = o; o += up256((size_t)BH * L.achunks * r * d * 4);
    L.Wp = o; o += up256((size_t)BH * r * d * 4);
    L.Xw = o; o += up256((size_t)BH * r * d * 4);
    L.dWm = o; o += up256((size_t)BH * r * d * 4);
    L.dbeta_direct = o; o += up256((size_t)BH * r * 4);
    for (int side = 0; side < 2; ++side) { L.zpart[side] = o; o += up256((size_t)BH * (L.achunks > L.gchunks ? L.achunks : L.gchunks) * r * d * 4); }
    L.total = o;
    return L;
}

// A call on the stored kernel whose workspace would pass kPartBytes runs its slices in parts one after the other: batch rows,
// or heads of one row.  Below that nothing is gained, a part of that size keeps the device busy for milliseconds.
constexpr size_t kPartBytes = (size_t)8 << 30;
struct Parts {
    int rows, heads;         // of a part; heads < H only with rows == 1
};
// bytes(rows, heads): workspace of such a part
template <typename F> Parts split_parts(int B, int H, F bytes)
{
    auto most = [](int n, auto fits) {                        // the largest k <= n that fits, then as even as the parts allow
        int lo = 1, hi = n;
        while (lo < hi) {
            const int mid = lo + (hi - lo + 1) / 2;
            if (fits(mid)) lo = mid; else hi = mid - 1;
        }
        const int parts = (n + lo - 1) / lo;
        return (n + parts - 1) / parts;
    };
    if (B < 1 || bytes(B, H) <= kPartBytes) return Parts{B, H};
    if (bytes(1, H) <= kPartBytes) return Parts{most(B, [&](int k) { return bytes(k, H) <= kPartBytes; }), H};
    return Parts{1, most(H, [&](int k) { return bytes(1, k) <= kPartBytes; })};
}
// Workspace of the whole call: that of a part or of the smaller last one.
template <typename F> size_t parts_bytes(int B, int H, F bytes)
{
    const Parts P = split_parts(B, H, bytes);
    size_t most = bytes(P.rows, P.heads);
    if (P.rows > 0 && B % P.rows != 0 && bytes(B % P.rows, H) > most) most = bytes(B % P.rows, H);
    if (H % P.heads != 0 && bytes(P.rows, H % P.heads) > most) most = bytes(P.rows, H % P.heads);
    return most;
}
// run(b0, rows, h0, heads) for every part, until one fails
template <typename F> cudaError_t for_parts(int B, int H, Parts P, F run)
{
    for (int b = 0; b < B; b += P.rows)
        for (int h = 0; h < H; h += P.heads) {
            const cudaError_t e = run(b, B - b < P.rows ? B - b : P.rows, h, H - h < P.heads ? H - h : P.heads);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

template <typename T> inline T *at(void *ws, size_t off) { return reinterpret_cast<T *>(static_cast<char *>(ws) + off); }

// bf16 tensors only: for float32 ones the interface has always asked for more than the kernel takes
Parts forward_parts(int B, int H, int nq, int nk, int d, int r, int dtype, bool variant)
{
    if (dtype == LOT_F32) return Parts{B, H};
    return split_parts(B, H, [&](int rows, int heads) { return forward_layout(rows, heads, nq, nk, d, r, dtype, variant).total; });
}
size_t forward_bytes(int B, int H, int nq, int nk, int d, int r, int dtype, bool variant)
{
    auto bytes = [&](int rows, int heads) { return forward_layout(rows, heads, nq, nk, d, r, dtype, variant).total; };
    return dtype == LOT_F32 ? bytes(B, H) : parts_bytes(B, H, bytes);
}
size_t bwd_bytes(int B, int H, int n, int d, int r, int iters)
{
    return parts_bytes(B, H, [&](int rows, int heads) { return bwd_sweep_layout(rows, heads, n, d, r, iters).total; });
}

struct Managed {
    void *ptr = nullptr;
    size_t bytes = 0;
};
Managed g_managed[kMaxDevices];
std::mutex g_managed_mu;

// Which path last ran on a workspace, and the tag of that call: the resident path keeps its status word tagged
// instead of clearing it, so reading it needs the tag (lot_device_status).
struct WsRecord {
    int path;
    unsigned tag;
    size_t fused_off;
};
std::unordered_map<const void *, WsRecord> g_ws_records;
std::mutex g_ws_mu;
void remember_ws(const void *ws, int path, unsigned tag, size_t fused_off)
{
    std::lock_guard<std::mutex> lock(g_ws_mu);
    if (g_ws_records.size() > 65536) g_ws_records.clear();
    g_ws_records[ws] = WsRecord{path, tag, fused_off};
}

enum { kPathGeneral = 0, kPathStreamed = 1, kPathResident = 2, kPathSlice = 3, kPathLong = 4 };
std::atomic<int> g_force_path{-1};      // test hook: 0 picks the general path, 1, 2 or 4 that tensor-core path wherever it can run
int choose_path(int dtype, int B, int H, int n, int d, int r, int iters)
{
    if (!fused_supported(dtype, d, r) || B < 1 || n < 1) return kPathGeneral;
    const bool res_ok = resident_geometry(dtype, B, H, n, d, r).ok;
    const bool slice_ok = slice_supported(dtype, n, d, r);
    const int force = g_force_path.load();
    if (force == kPathGeneral) return kPathGeneral;
    if (force == kPathStreamed) return kPathStreamed;
    if (force == kPathLong && r > 16) return kPathLong;
    if (force == kPathResident) return res_ok ? kPathResident : kPathStreamed;
    // short sequences: a pair of thread blocks per slice, everything on chip
    if (slice_ok) return kPathSlice;
    // Everything below measured on B200 at T = 10 unless said otherwise; us, in the order general / streamed / resident / long.
    // r <= 16: the general path's float32 kernel, 1.05 to 4.5 times the streamed kernel's speed everywhere.
    const long long rows = (long long)B * H * n, slices = (long long)B * H, sms = device_sm_count();
    if (r <= 16) return kPathGeneral;
    // r <= 32: it too with few rows or short sequences (16 slices of 8192 tokens 118 / 152, 192 of 1024 157 / 328), then the
    // streamed path, which does not wait for memory there (16 of 11000 177 / 167, 16 of 16384 230 / 210).  Both keep
    // float32 between the passes, which the long path's bf16 kernel does not (potentials to 8e-5 of eps instead of 2e-6), so
    // it is taken only where a bf16 kernel always has been: about one slice per SM, of up to 14 tiles, whose kernel the
    // resident path would keep on the SM (128 slices of 1400 tokens 159 / 165 / 159 / 122, of 1700 189 / 196 / 179 / 144).
    if (r <= 32) {
        if (n <= 1200 || rows <= 100000) return kPathGeneral;
        if (iters >= 3 && n <= 1792 && slices <= sms && 2 * slices >= sms) return kPathLong;
        return rows <= 160000 ? kPathGeneral : kPathStreamed;
    }
    // Above that the long path takes everything up to 300000 rows (n = 2048, 16 slices 73 / 114 / - / 64; n = 16384, 16 slices
    // streamed 190, long 180) and all short sequences (n = 1024, 512 slices: 461 / - / - / 301), in calls of three iterations and
    // more: one or two show that the streamed path's first pass is on float32 values (errors of the potentials at n = 4096 in
    // units of eps: 5e-6 against 1.3e-4 after one, 1.1e-4 against 1.3e-4 after two, 1.6e-4 on both after three).
    return iters >= 3 && (n <= 1200 || rows <= 300000) ? kPathLong : kPathStreamed;
}

size_t path_bytes(int path, int dtype, int B, int H, int n, int d, int r)
{
    if (path == kPathResident) return up256(resident_layout(B, H, n, d, r).total) + fused_layout(B, H, n, d, r).total;
    if (path == kPathStreamed) return fused_layout(B, H, n, d, r).total;
    if (path == kPathLong) return stream_plan(B * H, n).total;
    if (path == kPathSlice) return 256;                              // the status word
    return forward_bytes(B, H, n, n, d, r, dtype, false);
}

// Whether the first `bytes` of two tensors share memory.
bool overlap(const void *a, const void *b, size_t bytes)
{
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y ? y - x < bytes : x - y < bytes;
}

// A forward on the general path.
struct ForwardCall {
    const void *q, *k, *v;
    const float *z, *beta, *mass_q, *mass_k;
    int skip, terms;
    const int32_t *key_len;
    const float *g1_in, *g2_in;
    int dtype, B, H, nq, nk, d, r;
    float eps;
    int iters;
    void *out;
    float *g1_out, *g2_out;

    // heads h0 .. h0 + heads - 1 of batch rows b0 .. b0 + rows - 1, which are neighbours in memory
    ForwardCall part(int b0, int rows, int h0, int heads) const
    {
        ForwardCall c = *this;
        const size_t s = (size_t)b0 * H + h0, es = dtype == LOT_F32 ? 4 : 2;
        c.q = static_cast<const char *>(q) + s * nq * d * es; c.k = static_cast<const char *>(k) + s * nk * d * es;
        c.v = static_cast<const char *>(v) + s * nk * d * es; c.out = static_cast<char *>(out) + s * nq * d * es;
        c.z = z + (size_t)h0 * r * d; c.beta = beta + (size_t)h0 * r;
        if (mass_q) c.mass_q = mass_q + s * nq;
        if (mass_k) c.mass_k = mass_k + s * nk;
        if (key_len) c.key_len = key_len + b0;
        if (g1_in) c.g1_in = g1_in + s * r;
        if (g2_in) c.g2_in = g2_in + s * r;
        if (g1_out) c.g1_out = g1_out + s * r;
        if (g2_out) c.g2_out = g2_out + s * r;
        c.B = rows; c.H = heads;
        return c;
    }
};

// Both Sinkhorn problems and the apply stages.  first: of the call's parts (the status word is cleared once).
cudaError_t run_forward(const ForwardLayout &L, const ForwardCall &f, bool first, void *ws, cudaStream_t s)
{
    const int dtype = f.dtype, B = f.B, H = f.H, nq = f.nq, nk = f.nk, d = f.d, r = f.r, skip = f.skip, terms = f.terms, iters = f.iters;
    SweepArgs a{};
    SweepApplyArgs ap{};
    for (int side = 0; side < 2; ++side) {
        a.kt[side] = at<float>(ws, L.kt[side]); a.inv[side] = at<float>(ws, L.inv[side]);
        a.w[side] = at<float>(ws, L.w[side]); a.gref[side] = at<double>(ws, L.gref[side]);
        ap.kt[side] = a.kt[side]; ap.inv[side] = a.inv[side]; ap.w[side] = a.w[side];
    }
    a.x[0] = f.q; a.x[1] = f.k; a.z = f.z; a.beta = f.beta; a.key_len = f.key_len;
    a.mass[0] = f.mass_q; a.mass[1] = f.mass_k; a.g_in[0] = f.g1_in; a.g_in[1] = f.g2_in; a.g_out[0] = f.g1_out; a.g_out[1] = f.g2_out;
    a.xbuf = at<unsigned long long>(ws, L.xbuf); a.status = at<int>(ws, 0);
    a.head = at<uint4>(ws, first ? 0 : 256); a.head_words = (L.head_end - (first ? 0 : 256)) / 16;
    a.B = B; a.H = H; a.d = d; a.r = r; a.n[0] = nq; a.n[1] = nk; a.skip = skip; a.terms = terms;
    a.C = L.plan.C; a.K = L.plan.K; a.groups = L.plan.groups; a.srows = L.plan.srows; a.tcols = L.plan.tcols;
    a.scale = 1.4426950408889634 / (double)f.eps; a.eps_ln2 = (double)f.eps * 0.6931471805599453;
    a.iters = iters;
    cudaError_t e;
    if ((e = launch_build(L.plan.RP, a, dtype, s)) != cudaSuccess) return e;
    if ((e = launch_sweep(L.plan, a, dtype, s)) != cudaSuccess) return e;
    ap.beta = f.beta; ap.key_len = f.key_len; ap.mass2 = f.mass_k; ap.v = f.v; ap.out = f.out;
    ap.wpart = at<float>(ws, L.wpart); ap.Wp = at<float>(ws, L.Wp); ap.counter = at<unsigned>(ws, L.counter);
    ap.B = B; ap.H = H; ap.nq = nq; ap.nk = nk; ap.d = d; ap.r = r; ap.RP = L.plan.RP; ap.skip = skip; ap.terms = terms;
    ap.chunks = L.achunks; ap.rows_per_chunk = L.arows;
    if ((e = launch_sweep_apply_w(ap, dtype, s)) != cudaSuccess) return e;
    return launch_sweep_apply_out(ap, dtype, s);
}

// ... of all parts, the class-token row of each behind it.
cudaError_t run_forward_parts(const ForwardCall &f, bool variant, float cls_tau, void *ws, cudaStream_t s)
{
    return for_parts(f.B, f.H, forward_parts(f.B, f.H, f.nq, f.nk, f.d, f.r, f.dtype, variant), [&](int b0, int rows, int h0, int heads) {
        const ForwardCall c = f.part(b0, rows, h0, heads);
        const ForwardLayout L = forward_layout(rows, heads, f.nq, f.nk, f.d, f.r, f.dtype, variant);
        const cudaError_t e = run_forward(L, c, b0 == 0 && h0 == 0, ws, s);
        if (e != cudaSuccess || !f.skip) return e;
        return launch_cls_row(c.q, c.k, c.v, c.key_len, f.dtype, rows, heads, f.nq, f.nk, f.d, cls_tau, at<float>(ws, L.scores), c.out, s);
    });
}

// lot_attention_bwd for bf16 tensors, behind the argument checks.  first: of the call's parts; add: dz and dbeta hold the
// sums of earlier parts.
cudaError_t run_backward(const BwdSweepLayout &L, const void *q, const void *k, const void *v, const float *z, const float *beta,
                         const int32_t *key_len, const void *dout, int B, int H, int n, int d, int r, float eps, int iters, void *dq,
                         void *dk, void *dv, float *dz, float *dbeta, bool first, bool add, void *ws, cudaStream_t st)
{
    const int dt = LOT_BF16, RP = L.plan.RP;
    cudaError_t e;
    SweepBwdArgs b{};
    SweepArgs &a = b.s;
    SweepApplyArgs ap{};
    for (int side = 0; side < 2; ++side) {
        a.kt[side] = at<float>(ws, L.kt[side]); a.inv[side] = at<float>(ws, L.inv[side]);
        a.w[side] = at<float>(ws, L.w[side]); a.gref[side] = at<double>(ws, L.gref[side]);
        ap.kt[side] = a.kt[side]; ap.inv[side] = a.inv[side]; ap.w[side] = a.w[side];
        b.dC[side] = at<float>(ws, L.dC[side]);
        a.n[side] = n;
    }
    a.x[0] = q; a.x[1] = k; a.z = z; a.beta = beta; a.key_len = key_len;
    a.xbuf = at<unsigned long long>(ws, L.xbuf);
    a.hist = at<float>(ws, L.hist); a.hist_g = at<double>(ws, L.hist_g); a.wide = at<int>(ws, L.wide); a.status = at<int>(ws, 0);
    a.head = at<uint4>(ws, first ? 0 : 256); a.head_words = (L.head_end - (first ? 0 : 256)) / 16;
    a.B = B; a.H = H; a.d = d; a.r = r;
    a.C = L.plan.C; a.K = L.plan.K; a.groups = L.plan.groups; a.srows = L.plan.srows; a.tcols = L.plan.tcols;
    a.scale = 1.4426950408889634 / (double)eps; a.eps_ln2 = (double)eps * 0.6931471805599453;
    a.iters = iters; a.terms = 3;
    // ---- the forward, keeping the weights of every iteration
    if ((e = launch_build(RP, a, dt, st)) != cudaSuccess) return e;
    if ((e = launch_sweep(L.plan, a, dt, st)) != cudaSuccess) return e;
    ap.beta = beta; ap.key_len = key_len; ap.v = v;
    ap.wpart = at<float>(ws, L.wpart); ap.Wp = at<float>(ws, L.Wp); ap.counter = at<unsigned>(ws, L.counter);
    ap.B = B; ap.H = H; ap.nq = n; ap.nk = n; ap.d = d; ap.r = r; ap.RP = RP; ap.terms = 3;
    ap.chunks = L.achunks; ap.rows_per_chunk = L.arows;
    // W' = Diag(1/beta) Gamma2 V, and with it the reverse of the read-out, Eq. (4), out = R1 W': R1^T dout / (n beta) is the key-side
    // product on the query side
    SweepApplyArgs aq = ap;
    aq.kt[1] = ap.kt[0]; aq.inv[1] = ap.inv[0]; aq.w[1] = ap.w[0]; aq.key_len = nullptr; aq.v = dout; aq.Wp = at<float>(ws, L.Xw);
    aq.wpart = at<float>(ws, L.wpart2); aq.counter = at<unsigned>(ws, L.counter2);
    if ((e = launch_sweep_apply_w(ap, dt, st, &aq)) != cudaSuccess) return e;
    float *dbd = at<float>(ws, L.dbeta_direct), *dWm = at<float>(ws, L.dWm);
    if ((e = launch_bwd_w_fix(at<float>(ws, L.Xw), ap.Wp, key_len, dWm, dbd, B, H, n, d, r, st)) != cudaSuccess) return e;
    SweepApplyArgs av = ap;                                                             // dV = Gamma2 dW: the query-side product on the key side
    av.kt[0] = ap.kt[1]; av.inv[0] = ap.inv[1]; av.w[0] = ap.w[1]; av.Wp = dWm; av.out = dv; av.out_len = key_len;
    if ((e = launch_sweep_apply_out(av, dt, st)) != cudaSuccess) return e;
    b.g[0] = dout; b.g[1] = v; b.wmat[0] = ap.Wp; b.wmat[1] = dWm;
    b.coef = at<float2>(ws, L.coef); b.fk = at<float>(ws, L.fk); b.gpart = at<float>(ws, L.gpart); b.dbeta_acc = at<float>(ws, L.dbeta_acc);
    b.T = iters; b.tiles = L.tiles; b.eps = (double)eps;
    if ((e = launch_bwd_close(RP, b, st)) != cudaSuccess) return e;
    // ---- the iterations, last first
    a.seq0 = 4u * (unsigned)(iters + 1) * (unsigned)L.rounds;
    if ((e = launch_bwd_reverse(L.plan, b, st)) != cudaSuccess) return e;
    if (sweep_grad_supported(r, d)) {
        SweepGradArgs g{};
        g.b = b; g.dx[0] = dq; g.dx[1] = dk; g.chunks = L.gchunks; g.rows = L.grows;
        for (int side = 0; side < 2; ++side) g.part[side] = at<float>(ws, L.zpart[side]);
        if ((e = launch_sweep_grad(RP, g, st)) != cudaSuccess) return e;
        return launch_bwd_merge(g.part[0], g.part[1], dbd, b.dbeta_acc, dz, dbeta, B, H, d, r, RP, L.gchunks, add, st);
    }
    if (iters > 0 && (e = launch_bwd_assemble(RP, b, st)) != cudaSuccess) return e;
    // ---- C = X Z^T: dX = dC Z, dZ = dC^T X, the same two products with the gradient in place of the plan
    for (int side = 0; side < 2; ++side) {
        SweepApplyArgs x = ap;
        x.kt[0] = b.dC[side]; x.inv[0] = nullptr; x.w[0] = nullptr; x.Wp = const_cast<float *>(z); x.per_head = 1;
        x.out = side ? dk : dq; x.out_len = side ? key_len : nullptr;
        if ((e = launch_sweep_apply_out(x, dt, st)) != cudaSuccess) return e;
        SweepApplyArgs y = ap;
        y.kt[1] = b.dC[side]; y.inv[1] = nullptr; y.w[1] = nullptr; y.beta = nullptr; y.key_len = side ? key_len : nullptr;
        y.v = side ? k : q; y.Wp = nullptr; y.wpart = at<float>(ws, L.zpart[side]);
        if ((e = launch_sweep_apply_w(y, dt, st)) != cudaSuccess) return e;
    }
    return launch_bwd_merge(at<float>(ws, L.zpart[0]), at<float>(ws, L.zpart[1]), dbd, b.dbeta_acc, dz, dbeta, B, H, d, r, RP, L.achunks, add, st);
}

// Scratch of lot_sinkhorn_static: part of the library image, present on every device that loads
// it.  In host code this name is only a handle for cudaGetSymbolAddress, never a device address.
static __device__ __align__(256) unsigned char g_static_scratch[LOT_STATIC_SCRATCH_BYTES];
void *g_static_ptr[kMaxDevices];   // device address of the array, per device (looked up once)
std::mutex g_static_mu;

} // namespace

extern "C" {

#ifdef LOT_DEBUG
int lot_version(void) { return 100 + 100000; }      // the bounds-check build answers 100100
#else
int lot_version(void) { return 100; }
#endif

const char *lot_status_string(int status)
{
    switch (status) {
    case LOT_OK: return "LOT_OK";
    case LOT_ERR_INVALID_ARG: return "LOT_ERR_INVALID_ARG: null or misaligned pointer, eps <= 0, iters < 0 or unknown dtype";
    case LOT_ERR_UNSUPPORTED_SHAPE: return "LOT_ERR_UNSUPPORTED_SHAPE: need 1 <= r <= 256, 8 <= d <= 256, d % 8 == 0, B*H <= 32767, n*r and n*d < 2^31";
    case LOT_ERR_WORKSPACE: return "LOT_ERR_WORKSPACE: workspace null, not 256-byte aligned or too small (lot_sinkhorn_static: the problem needs more than LOT_STATIC_SCRATCH_BYTES)";
    case LOT_ERR_CUDA: return "LOT_ERR_CUDA: a CUDA runtime call or kernel launch failed";
    default: return "unknown lot status";
    }
}

int lot_cost(const void *x, const float *z, int dtype, int B, int H, int n, int d, int r,
             float *cost, lot_stream_t stream)
{
    if (dtype != LOT_F32 && dtype != LOT_BF16) return LOT_ERR_INVALID_ARG;
    int st = check_dims(B, H, n, r);
    if (st != LOT_OK) return st;
    st = check_d(n, d);
    if (st != LOT_OK) return st;
    if (B == 0 || n == 0) return LOT_OK;
    if (!x || !z || !cost) return LOT_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(z) || !aligned16(cost)) return LOT_ERR_INVALID_ARG;
    cudaError_t e = launch_cost(x, z, dtype, B * H, H, n, d, r, cost, false, (cudaStream_t)stream);
    return e == cudaSuccess ? LOT_OK : LOT_ERR_CUDA;
}

size_t lot_sinkhorn_workspace_bytes(int B, int H, int n, int r)
{
    if (check_dims(B, H, n, r) != LOT_OK) return 0;
    return sink_layout(B * H, n, r, 0, 8).total;
}

int lot_sinkhorn(const float *cost, const float *beta, const int32_t *len,
                 int B, int H, int n, int r, float eps, int iters,
                 float *g, float *f, float *plan,
                 void *ws, size_t ws_bytes, lot_stream_t stream)
{
    int st = check_dims(B, H, n, r);
    if (st != LOT_OK) return st;
    if (!(eps > 0.f) || !isfinite(eps) || iters < 0) return LOT_ERR_INVALID_ARG;
    if (B == 0 || n == 0) return LOT_OK;
    if (!cost || !beta || !g) return LOT_ERR_INVALID_ARG;
    if (!aligned16(cost) || !aligned16(beta) || !aligned16(g) || !aligned16(f) || !aligned16(plan) ||
        (len && (reinterpret_cast<uintptr_t>(len) & 3u)))
        return LOT_ERR_INVALID_ARG;
    const int nprob = B * H;
    SinkLayout L = sink_layout(nprob, n, r, 0, 8);
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < L.total) return LOT_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemsetAsync(ws, 0, L.head_end, s) != cudaSuccess) return LOT_ERR_CUDA;

    PassArgs a{};
    a.cost = cost; a.beta = beta; a.len = len; a.len_from = 0;
    a.G = at<void>(ws, L.G); a.part = at<float>(ws, L.part); a.counter = at<unsigned>(ws, L.counter);
    a.M = at<void>(ws, L.M); a.g_out = g; a.f_out = f; a.plan_out = plan;
    a.status = at<int>(ws, L.status);
    a.nprob = nprob; a.B = B; a.H = H; a.n = n; a.r = r;
    a.chunks = L.chunks; a.rows_per_chunk = L.rows_per_chunk;
    a.mode = kModeCostF32Wide;
    a.scale_d = 1.4426950408889634 / (double)eps;
    a.eps_ln2 = (float)((double)eps * 0.6931471805599453);
    for (int it = 0; it < iters; ++it)
        if (launch_sinkhorn_pass(a, false, s) != cudaSuccess) return LOT_ERR_CUDA;
    if (launch_sinkhorn_pass(a, true, s) != cudaSuccess) return LOT_ERR_CUDA;
    return LOT_OK;
}

int lot_sinkhorn_static(const float *cost, const float *beta, const int32_t *len,
                        int B, int H, int n, int r, float eps, int iters,
                        float *g, float *f, float *plan, int32_t *status_out,
                        lot_stream_t stream)
{
    // every argument check comes first, in lot_sinkhorn's order, so that a bad call is refused before any device work
    int st = check_dims(B, H, n, r);
    if (st != LOT_OK) return st;
    if (!(eps > 0.f) || !isfinite(eps) || iters < 0) return LOT_ERR_INVALID_ARG;
    if (status_out && (reinterpret_cast<uintptr_t>(status_out) & 3u)) return LOT_ERR_INVALID_ARG;
    if (B == 0 || n == 0) return LOT_OK;
    if (!cost || !beta || !g) return LOT_ERR_INVALID_ARG;
    if (!aligned16(cost) || !aligned16(beta) || !aligned16(g) || !aligned16(f) || !aligned16(plan) ||
        (len && (reinterpret_cast<uintptr_t>(len) & 3u)))
        return LOT_ERR_INVALID_ARG;
    if (sink_layout(B * H, n, r, 0, 8).total > (size_t)LOT_STATIC_SCRATCH_BYTES) return LOT_ERR_WORKSPACE;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return LOT_ERR_CUDA;
    void *ws = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (g_static_ptr[dev] == nullptr) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || p == nullptr) {
                (void)cudaGetLastError();
                return LOT_ERR_CUDA;
            }
            g_static_ptr[dev] = p;
        }
        ws = g_static_ptr[dev];
    }
    st = lot_sinkhorn(cost, beta, len, B, H, n, r, eps, iters, g, f, plan, ws, LOT_STATIC_SCRATCH_BYTES, stream);
    if (st != LOT_OK) return st;
    if (status_out && cudaMemcpyAsync(status_out, ws, sizeof(int32_t), cudaMemcpyDeviceToDevice,
                                      (cudaStream_t)stream) != cudaSuccess)
        return LOT_ERR_CUDA;
    return LOT_OK;
}

size_t lot_workspace_bytes(int B, int H, int n, int d, int r, int dtype)
{
    if (dtype != LOT_F32 && dtype != LOT_BF16) return 0;
    if (check_dims(B, H, n, r) != LOT_OK || check_d(n, d) != LOT_OK) return 0;
    // the most of any number of iterations
    const size_t few = path_bytes(choose_path(dtype, B, H, n, d, r, 0), dtype, B, H, n, d, r);
    const size_t many = path_bytes(choose_path(dtype, B, H, n, d, r, 1 << 20), dtype, B, H, n, d, r);
    return few > many ? few : many;
}

int lot_path(int dtype, int B, int H, int n, int d, int r, int iters)
{
    if (dtype != LOT_F32 && dtype != LOT_BF16) return 0;
    if (check_dims(B, H, n, r) != LOT_OK || check_d(n, d) != LOT_OK) return 0;
    return choose_path(dtype, B, H, n, d, r, iters);
}

int lot_launch_count(int dtype, int B, int H, int n, int d, int r, int iters)
{
    if (iters < 0) return 0;
    const int path = lot_path(dtype, B, H, n, d, r, iters);
    if (path == kPathResident) return 1 + 2;                        // the two streamed kernels return at once unless asked to redo
    if (path == kPathStreamed) return fused_launches(B, H, n, r, iters);
    if (path == kPathSlice) return 1;
    if (path == kPathLong) return 3;
    if (B < 1 || n < 1) return 0;
    const Parts P = forward_parts(B, H, n, n, d, r, dtype, false);
    return 4 * ((B + P.rows - 1) / P.rows) * ((H + P.heads - 1) / P.heads);
}

int lot_debug_hook(int what, long long value)
{
    if (what < 1 || what > 4) return LOT_ERR_INVALID_ARG;
    if (what == 4) g_force_path.store((int)value);
    else resident_debug(what, value);
    return LOT_OK;
}

int lot_attention_fwd_ex(const void *q, const void *k, const void *v,
                         const float *z, const float *beta, const int32_t *key_len,
                         int dtype, int B, int H, int n, int d, int r, float eps, int iters,
                         void *out, float *g1_out, float *g2_out,
                         void *ws, size_t ws_bytes, lot_stream_t stream)
{
    if (dtype != LOT_F32 && dtype != LOT_BF16) return LOT_ERR_INVALID_ARG;
    int st = check_dims(B, H, n, r);
    if (st != LOT_OK) return st;
    st = check_d(n, d);
    if (st != LOT_OK) return st;
    if (!(eps > 0.f) || !isfinite(eps) || iters < 0) return LOT_ERR_INVALID_ARG;
    if (B == 0 || n == 0) return LOT_OK;
    if (!q || !k || !v || !z || !beta || !out) return LOT_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(z) || !aligned16(beta) ||
        !aligned16(out) || !aligned16(g1_out) || !aligned16(g2_out) ||
        (key_len && (reinterpret_cast<uintptr_t>(key_len) & 3u)))
        return LOT_ERR_INVALID_ARG;
    int path = choose_path(dtype, B, H, n, d, r, iters);
    // the long path keeps part of the kernel in out until it is written; the streamed one takes an output over an input
    const size_t bytes = (size_t)B * H * n * d * 2;
    if (path == kPathLong && (overlap(out, q, bytes) || overlap(out, k, bytes) || overlap(out, v, bytes))) path = kPathStreamed;
    if (path == kPathSlice) {
        if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < 256) return LOT_ERR_WORKSPACE;
        remember_ws(ws, kPathSlice, 0, 0);
        cudaError_t e = slice_attention(q, k, v, z, beta, key_len, B, H, n, r, eps, iters, out, g1_out, g2_out,
                                        at<int>(ws, 0), (cudaStream_t)stream);
        return e == cudaSuccess ? LOT_OK : LOT_ERR_CUDA;
    }
    if (path == kPathLong) {
        if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < stream_plan(B * H, n).total) return LOT_ERR_WORKSPACE;
        remember_ws(ws, kPathLong, 0, 0);
        return stream_attention(q, k, v, z, beta, key_len, B, H, n, r, eps, iters, out, g1_out, g2_out, ws, (cudaStream_t)stream) == cudaSuccess
                   ? LOT_OK : LOT_ERR_CUDA;
    }
    if (path != kPathGeneral) {
        const size_t res_bytes = path == kPathResident ? up256(resident_layout(B, H, n, d, r).total) : 0;
        const size_t need = res_bytes + fused_layout(B, H, n, d, r).total;
        if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < need) return LOT_ERR_WORKSPACE;
        cudaStream_t s = (cudaStream_t)stream;
        unsigned tag = 0;
        const unsigned *redo = nullptr;
        if (path == kPathResident) {
            if (resident_attention(q, k, v, z, beta, key_len, B, H, n, d, r, eps, iters, out, g1_out, g2_out, ws, &tag, s) !=
                cudaSuccess) {
                (void)cudaGetLastError();
                return LOT_ERR_CUDA;
            }
            redo = at<unsigned>(ws, resident_layout(B, H, n, d, r).status + 8);
        }
        remember_ws(ws, path, tag, res_bytes);
        // behind a resident launch the streamed kernels run only if that launch asked for it (a problem outside the
        // range of the stored bf16 kernel); alone they are the path
        cudaError_t e = fused_attention(q, k, v, z, beta, key_len, B, H, n, d, r, eps, iters, out, g1_out, g2_out,
                                        at<char>(ws, res_bytes), redo, tag, s);
        return e == cudaSuccess ? LOT_OK : LOT_ERR_CUDA;
    }
    remember_ws(ws, kPathGeneral, 0, 0);
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < forward_bytes(B, H, n, n, d, r, dtype, false)) return LOT_ERR_WORKSPACE;
    // sizes of the tensor-core paths keep their hi + lo operands here too; a forced general path is float32 throughout
    const int terms = fused_supported(dtype, d, r) && g_force_path.load() != kPathGeneral ? 2 : 3;
    const ForwardCall f{q, k, v, z, beta, nullptr, nullptr, 0, terms, key_len, nullptr, nullptr, dtype, B, H, n, n, d, r, eps, iters, out,
                        g1_out, g2_out};
    return run_forward_parts(f, false, 0.f, ws, (cudaStream_t)stream) == cudaSuccess ? LOT_OK : LOT_ERR_CUDA;
}

size_t lot_var_workspace_bytes(int B, int H, int nq, int nk, int d, int r, int dtype)
{
    if (dtype != LOT_F32 && dtype != LOT_BF16) return 0;
    if (check_dims(B, H, nq, r) != LOT_OK || check_dims(B, H, nk, r) != LOT_OK) return 0;
    if (check_d(nq, d) != LOT_OK || check_d(nk, d) != LOT_OK) return 0;
    return forward_bytes(B, H, nq, nk, d, r, dtype, true);
}

int lot_attention_fwd_var(const void *q, const void *k, const void *v, const float *z, const float *beta,
                          const float *a, const float *b, const int32_t *key_len,
                          const float *g1_in, const float *g2_in, int cls, float cls_tau,
                          int dtype, int B, int H, int nq, int nk, int d, int r, float eps, int iters,
                          void *out, float *g1_out, float *g2_out,
                          void *ws, size_t ws_bytes, lot_stream_t stream)
{
    if (dtype != LOT_F32 && dtype != LOT_BF16) return LOT_ERR_INVALID_ARG;
    int st = check_dims(B, H, nq, r);
    if (st == LOT_OK) st = check_dims(B, H, nk, r);
    if (st == LOT_OK) st = check_d(nq, d);
    if (st == LOT_OK) st = check_d(nk, d);
    if (st != LOT_OK) return st;
    if (!(eps > 0.f) || !isfinite(eps) || iters < 0) return LOT_ERR_INVALID_ARG;
    if (cls != 0 && cls != 1) return LOT_ERR_INVALID_ARG;
    if (cls && (!(cls_tau > 0.f) || !isfinite(cls_tau) || a != nullptr || b != nullptr)) return LOT_ERR_INVALID_ARG;
    if (B == 0 || nq == 0) return LOT_OK;
    if (nk == 0) return LOT_ERR_INVALID_ARG;
    if (!q || !k || !v || !z || !beta || !out) return LOT_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(z) || !aligned16(beta) || !aligned16(out) ||
        !aligned16(g1_out) || !aligned16(g2_out) || !aligned16(g1_in) || !aligned16(g2_in) || !aligned16(a) ||
        !aligned16(b) || (key_len && (reinterpret_cast<uintptr_t>(key_len) & 3u)))
        return LOT_ERR_INVALID_ARG;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < forward_bytes(B, H, nq, nk, d, r, dtype, true)) return LOT_ERR_WORKSPACE;
    remember_ws(ws, kPathGeneral, 0, 0);
    // the class token is neither a query nor a key of the transport problem: it is skipped on both sides
    const ForwardCall f{q, k, v, z, beta, a, b, cls, 3, key_len, g1_in, g2_in, dtype, B, H, nq, nk, d, r, eps, iters, out, g1_out, g2_out};
    return run_forward_parts(f, true, cls_tau, ws, (cudaStream_t)stream) == cudaSuccess ? LOT_OK : LOT_ERR_CUDA;
}

int lot_attention_fwd(const float *q, const float *k, const float *v,
                      const float *z, const float *beta,
                      int B, int H, int n, int d, int r, float eps, int iters,
                      float *out, lot_stream_t stream)
{
    int st = check_dims(B, H, n, r);
    if (st != LOT_OK) return st;
    st = check_d(n, d);
    if (st != LOT_OK) return st;
    if (B == 0 || n == 0) return LOT_OK;
    const size_t need = forward_layout(B, H, n, n, d, r, LOT_F32, false).total;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return LOT_ERR_CUDA;
    void *ws = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_managed_mu);
        Managed &m = g_managed[dev];
        if (m.bytes < need) {
            if (cudaDeviceSynchronize() != cudaSuccess) return LOT_ERR_CUDA;
            if (m.ptr) cudaFree(m.ptr);
            m.ptr = nullptr; m.bytes = 0;
            if (cudaMalloc(&m.ptr, need) != cudaSuccess) { (void)cudaGetLastError(); m.ptr = nullptr; return LOT_ERR_CUDA; }
            m.bytes = need;
        }
        ws = m.ptr;
    }
    return lot_attention_fwd_ex(q, k, v, z, beta, nullptr, LOT_F32, B, H, n, d, r, eps, iters,
                                out, nullptr, nullptr, ws, need, stream);
}

int lot_device_status(const void *ws, lot_stream_t stream, int *status)
{
    if (!status) return LOT_ERR_INVALID_ARG;
    if (!ws) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return LOT_ERR_CUDA;
        std::lock_guard<std::mutex> lock(g_managed_mu);
        ws = g_managed[dev].ptr;
        if (!ws) { *status = 0; return LOT_OK; }
    }
    cudaStream_t s = (cudaStream_t)stream;
    WsRecord rec{kPathGeneral, 0, 0};
    {
        std::lock_guard<std::mutex> lock(g_ws_mu);
        auto it = g_ws_records.find(ws);
        if (it != g_ws_records.end()) rec = it->second;
    }
    if (rec.path != kPathResident) {
        if (cudaMemcpyAsync(status, ws, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return LOT_ERR_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return LOT_ERR_CUDA;
        if (kernels_debug_flag() | backward_debug_flag()) *status |= LOT_DEV_BOUNDS;      // bounds-check build only
        return LOT_OK;
    }
    // resident path: {flags | tag << 32, redo word} at the start, the streamed kernels' word behind the resident block
    unsigned head[4] = {0, 0, 0, 0};
    int streamed = 0;
    if (cudaMemcpyAsync(head, ws, sizeof(head), cudaMemcpyDeviceToHost, s) != cudaSuccess) return LOT_ERR_CUDA;
    if (cudaMemcpyAsync(&streamed, static_cast<const char *>(ws) + rec.fused_off, sizeof(int), cudaMemcpyDeviceToHost, s) !=
        cudaSuccess)
        return LOT_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return LOT_ERR_CUDA;
    const int mine = head[1] == rec.tag ? (int)head[0] : 0;
    // a call that was recomputed reports the recomputation's flags (and a timeout of the first attempt, if any)
    *status = head[2] == rec.tag ? (LOT_DEV_RECOMPUTED | streamed | (mine & LOT_DEV_TIMEOUT)) : (mine | streamed);
    return LOT_OK;
}

size_t lot_bwd_workspace_bytes(int B, int H, int n, int d, int r, int dtype, int iters)
{
    if (dtype != LOT_F32 && dtype != LOT_BF16) return 0;
    if (check_dims(B, H, n, r) != LOT_OK || check_d(n, d) != LOT_OK || iters < 0) return 0;
    return dtype == LOT_BF16 ? bwd_bytes(B, H, n, d, r, iters) : bwd_layout(B, H, n, d, r, iters).total;
}

int lot_attention_bwd(const void *q, const void *k, const void *v, const float *z, const float *beta,
                      const int32_t *key_len, const void *dout,
                      int dtype, int B, int H, int n, int d, int r, float eps, int iters,
                      void *dq, void *dk, void *dv, float *dz, float *dbeta,
                      void *ws, size_t ws_bytes, lot_stream_t stream)
{
    if (dtype != LOT_F32 && dtype != LOT_BF16) return LOT_ERR_INVALID_ARG;
    int st = check_dims(B, H, n, r);
    if (st != LOT_OK) return st;
    st = check_d(n, d);
    if (st != LOT_OK) return st;
    if (!(eps > 0.f) || !isfinite(eps) || iters < 0) return LOT_ERR_INVALID_ARG;
    if (!z || !beta || !dz || !dbeta) return LOT_ERR_INVALID_ARG;
    if (!aligned16(z) || !aligned16(beta) || !aligned16(dz) || !aligned16(dbeta)) return LOT_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (B == 0 || n == 0) {
        // no tokens: the pivots receive no gradient
        if (cudaMemsetAsync(dz, 0, (size_t)H * r * d * sizeof(float), s) != cudaSuccess) return LOT_ERR_CUDA;
        if (cudaMemsetAsync(dbeta, 0, (size_t)H * r * sizeof(float), s) != cudaSuccess) return LOT_ERR_CUDA;
        return LOT_OK;
    }
    if (!q || !k || !v || !dout || !dq || !dk || !dv) return LOT_ERR_INVALID_ARG;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(dout) || !aligned16(dq) || !aligned16(dk) ||
        !aligned16(dv) || (key_len && (reinterpret_cast<uintptr_t>(key_len) & 3u)))
        return LOT_ERR_INVALID_ARG;
    if (dtype == LOT_BF16) {
        if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < bwd_bytes(B, H, n, d, r, iters)) return LOT_ERR_WORKSPACE;
        remember_ws(ws, kPathGeneral, 0, 0);
        const Parts P = split_parts(B, H, [&](int rows, int heads) { return bwd_sweep_layout(rows, heads, n, d, r, iters).total; });
        return for_parts(B, H, P, [&](int b0, int rows, int h0, int heads) {
            const size_t o = ((size_t)b0 * H + h0) * n * d * 2, oz = (size_t)h0 * r * d, ob = (size_t)h0 * r;
            auto in = [&](const void *p) { return static_cast<const void *>(static_cast<const char *>(p) + o); };
            auto res = [&](void *p) { return static_cast<void *>(static_cast<char *>(p) + o); };
            return run_backward(bwd_sweep_layout(rows, heads, n, d, r, iters), in(q), in(k), in(v), z + oz, beta + ob,
                                key_len ? key_len + b0 : nullptr, in(dout), rows, heads, n, d, r, eps, iters, res(dq), res(dk), res(dv),
                                dz + oz, dbeta + ob, b0 == 0 && h0 == 0, b0 > 0, ws, s);
        }) == cudaSuccess ? LOT_OK : LOT_ERR_CUDA;
    }
    const BwdLayout L = bwd_layout(B, H, n, d, r, iters);
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < L.total) return LOT_ERR_WORKSPACE;
    remember_ws(ws, kPathGeneral, 0, 0);
    const size_t lt = 8;
    const int BH = B * H, np = 2 * BH;
    if (cudaMemsetAsync(ws, 0, L.head_end, s) != cudaSuccess) return LOT_ERR_CUDA;

    // ---- the forward, keeping the potentials of every iteration
    char *cost1 = at<char>(ws, L.cost);
    char *cost2 = cost1 + (size_t)BH * n * r * lt;
    if (launch_cost(q, z, dtype, BH, H, n, d, r, cost1, true, s) != cudaSuccess) return LOT_ERR_CUDA;
    if (launch_cost(k, z, dtype, BH, H, n, d, r, cost2, true, s) != cudaSuccess) return LOT_ERR_CUDA;
    char *hist = at<char>(ws, L.hist);
    const size_t hstep = (size_t)np * r * lt;
    PassArgs a{};
    a.cost = cost1; a.beta = beta; a.len = key_len; a.len_from = BH;
    a.part = at<float>(ws, L.part); a.counter = at<unsigned>(ws, L.counter);
    a.M = at<void>(ws, L.M); a.status = at<int>(ws, 0);
    a.nprob = np; a.B = B; a.H = H; a.n = n; a.r = r;
    a.chunks = L.chunks; a.rows_per_chunk = L.rows_per_chunk;
    a.mode = kModeWide;
    a.scale_d = 1.4426950408889634 / (double)eps;
    a.eps_ln2 = (float)((double)eps * 0.6931471805599453);
    for (int it = 0; it < iters; ++it) {
        a.G = hist + (size_t)it * hstep; a.G_next = hist + (size_t)(it + 1) * hstep;
        if (launch_sinkhorn_pass(a, false, s) != cudaSuccess) return LOT_ERR_CUDA;
    }
    char *Gfin = hist + (size_t)iters * hstep;
    a.G = Gfin; a.G_next = nullptr;
    if (launch_sinkhorn_pass(a, true, s) != cudaSuccess) return LOT_ERR_CUDA;

    char *M1 = at<char>(ws, L.M), *M2 = M1 + (size_t)BH * n * lt;
    char *G1 = Gfin, *G2 = Gfin + (size_t)BH * r * lt;
    float *Wp = at<float>(ws, L.Wp), *Xw = at<float>(ws, L.Xw), *dWm = at<float>(ws, L.dWm);
    ApplyArgs ap{};
    ap.cost1 = cost1; ap.cost2 = cost2; ap.G1 = G1; ap.G2 = G2; ap.M1 = M1; ap.M2 = M2;
    ap.beta = beta; ap.key_len = key_len; ap.v = v; ap.out = nullptr;
    ap.wpart = at<float>(ws, L.wpart); ap.Wp = Wp; ap.counter = at<unsigned>(ws, L.counter2);
    ap.B = B; ap.H = H; ap.n = n; ap.nk = n; ap.d = d; ap.r = r;
    ap.chunks = L.achunks; ap.rows_per_chunk = L.arows; ap.scale_d = a.scale_d;
    if (launch_apply_w(ap, s) != cudaSuccess) return LOT_ERR_CUDA;                 // W' = Diag(1/beta) Gamma2 V

    // ---- reverse of the read-out, Eq. (4): out = R1 W'
    ApplyArgs aq = ap;                                  // R1^T dout / (n beta): the key-side kernel on the query side
    aq.cost2 = cost1; aq.G2 = G1; aq.M2 = M1; aq.key_len = nullptr; aq.v = dout; aq.Wp = Xw;
    if (launch_apply_w(aq, s) != cudaSuccess) return LOT_ERR_CUDA;
    float *dbd = at<float>(ws, L.dbeta_direct);
    if (launch_bwd_w_fix(Xw, Wp, key_len, dWm, dbd, B, H, n, d, r, s) != cudaSuccess) return LOT_ERR_CUDA;
    ApplyArgs av = ap;                                  // dV = Gamma2 dW: the query-side kernel on the key side
    av.cost1 = cost2; av.G1 = G2; av.M1 = M2; av.Wp = dWm; av.out = dv;
    if (launch_apply_out(av, s) != cudaSuccess) return LOT_ERR_CUDA;
    char *dC1 = at<char>(ws, L.dC);
    char *dC2 = dC1 + (size_t)BH * n * r * lt;
    if (launch_gemm_nt(dout, false, Wp, false, dC1, true, BH, H, n, d, r, s) != cudaSuccess) return LOT_ERR_CUDA;
    if (launch_gemm_nt(v, false, dWm, false, dC2, true, BH, H, n, d, r, s) != cudaSuccess) return LOT_ERR_CUDA;

    // ---- reverse of the closing token update, then of the iterations, last first
    BwdRowArgs br{};
    br.cost = cost1; br.dC = dC1; br.gamma = at<void>(ws, L.gamma); br.dbeta_acc = at<void>(ws, L.dbeta_acc);
    br.beta = beta; br.len = key_len; br.len_from = BH;
    br.part = at<void>(ws, L.part); br.counter = at<unsigned>(ws, L.counter);
    br.nprob = np; br.B = B; br.H = H; br.n = n; br.r = r;
    br.chunks = L.chunks; br.rows_per_chunk = L.rows_per_chunk;
    br.scale_d = a.scale_d; br.eps = (double)eps;
    br.Ga = Gfin; br.Gb = nullptr;
    if (launch_bwd_rows(br, true, s) != cudaSuccess) return LOT_ERR_CUDA;
    for (int it = iters; it >= 1; --it) {
        br.Ga = hist + (size_t)(it - 1) * hstep; br.Gb = hist + (size_t)it * hstep;
        if (launch_bwd_rows(br, false, s) != cudaSuccess) return LOT_ERR_CUDA;
    }

    // ---- C = X Z^T: dX = dC Z, dZ = dC^T X
    float *zt = at<float>(ws, L.zt);
    if (launch_transpose_z(z, zt, H, r, d, s) != cudaSuccess) return LOT_ERR_CUDA;
    if (launch_gemm_nt(dC1, true, zt, true, dq, false, BH, H, n, r, d, s) != cudaSuccess) return LOT_ERR_CUDA;
    if (launch_gemm_nt(dC2, true, zt, true, dk, false, BH, H, n, r, d, s) != cudaSuccess) return LOT_ERR_CUDA;
    if (launch_bwd_dz(dC1, q, k, at<void>(ws, L.dzpart), dbd, br.dbeta_acc, dz, dbeta, B, H, n, d, r, L.dzchunks, s) != cudaSuccess)
        return LOT_ERR_CUDA;
    return LOT_OK;
}

} // extern "C"
