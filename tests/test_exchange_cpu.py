"""The exchange of column sums between the blocks of a group, the code of group_columns itself, compiled for the host: a thread per GPU
thread, barriers that count arrivals and bytes as the hardware's do, and words in memory.  Totals are right in every block; where a
block's messages are dropped every wait ends, the call is flagged, and no barrier is armed while its phase is still open (which
would leave its count undefined)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CORE = os.path.join(ROOT, "paper_2509_23436_b200", "csrc", "lot_sweep_core.cuh")

FAKES = r"""
#include <pthread.h>
#include <sched.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <time.h>
#include <math.h>
#include <mutex>
#include <thread>
#include <vector>
#define __host__
#define __device__
#define __forceinline__ inline
typedef unsigned long long u64;
constexpr int kPeers = 8, kWords = 16;
static u64 kWaitNs;
static std::recursive_mutex mu;
typedef std::lock_guard<std::recursive_mutex> Hold;
struct Dim { int x; };
static thread_local Dim threadIdx;
static thread_local int g_block, g_cluster;                // the thread's block, and the first one of its cluster
static thread_local bool g_dropped;                        // its messages get lost
static int g_armed_open, g_lost;
struct Bar { int pending = 1, tx = 0; unsigned done = 0; };
static uint8_t g_mem[32][1 << 14];
static Bar g_bar[32][2];
constexpr uint32_t kBars = 1 << 13;                        // address of a block's barriers; block b's memory starts at b << 14
static Bar &bar_of(uint32_t a) { return g_bar[a >> 14][(a & 15) / 8]; }
static void settle(Bar &b) { if (b.pending == 0 && b.tx == 0) { b.pending = 1; ++b.done; } }
namespace sm100 {
static void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    Hold h(mu);
    Bar &b = bar_of(bar);
    if (b.pending == 0) { ++g_armed_open; return; }
    b.tx += bytes; --b.pending;
    settle(b);
}
}
static float neg_inf() { return -INFINITY; }
static unsigned __float_as_uint(float v) { unsigned u; memcpy(&u, &v, 4); return u; }
static float __uint_as_float(unsigned u) { float v; memcpy(&v, &u, 4); return v; }
static int __clz(int v) { return __builtin_clz(v); }
static void atomicOr(int *p, int v) { Hold h(mu); *p |= v; }
static u64 global_timer_ns() { sched_yield(); timespec t; clock_gettime(CLOCK_MONOTONIC, &t); return t.tv_sec * 1000000000ull + t.tv_nsec; }
static float lds(uint32_t a) { Hold h(mu); float v; memcpy(&v, g_mem[a >> 14] + (a & 16383), 4); return v; }
static uint32_t in_peer(uint32_t a, int o) { return (a & 16383) + ((uint32_t)(g_cluster + o) << 14); }
static void send(uint32_t dst, float v, uint32_t bar)
{
    Hold h(mu);
    if (g_dropped) { ++g_lost; return; }
    memcpy(g_mem[dst >> 14] + (dst & 16383), &v, 4);
    Bar &b = bar_of(bar);
    b.tx -= 4;
    settle(b);
}
static bool sends_arrived(uint32_t bar, unsigned parity) { Hold h(mu); return (bar_of(bar).done & 1) != parity; }
static void put_word(u64 *p, float v, unsigned tag)
{
    Hold h(mu);
    if (g_dropped) { ++g_lost; return; }
    *p = (u64)tag << 32 | __float_as_uint(v);
}
static u64 peek_word(const u64 *p) { Hold h(mu); return *p; }
struct Shared { volatile int *flag; uint32_t bars, peers; };
struct Args { int C, K; unsigned seq0; int *status; u64 *xbuf; };
"""

MAIN = r"""
constexpr int RP = 16, N = 12;
int main(int argc, char **argv)
{
    const int C = atoi(argv[1]), K = atoi(argv[2]), drop = atoi(argv[3]), from = atoi(argv[4]);
    kWaitNs = drop < 0 ? 60000000000ull : 200000000ull;
    std::vector<u64> words(2 * (C / K) * RP, 0);
    int status = 0, wrong = 0, flags[32] = {};
    Args a = {C, K, 0, &status, words.data()};
    pthread_barrier_t sync[32];
    std::vector<std::thread> all;
    for (int c = 0; c < C; ++c) {
        pthread_barrier_init(&sync[c], nullptr, RP);
        for (int b = 0; b < 2 && K > 1; ++b) sm100::mbar_arrive_expect_tx((c << 14) + kBars + 8 * b, peer_bytes(RP, C, K) / 2);
    }
    for (int c = 0; c < C; ++c)
        for (int t = 0; t < RP; ++t)
            all.emplace_back([&, c, t] {
                threadIdx.x = t; g_block = c; g_cluster = c / K * K;
                Shared S = {&flags[c], (uint32_t)(c << 14) + kBars, (uint32_t)c << 14};
                unsigned seq = 0;
                for (int i = 0; i < N; ++i) {
                    g_dropped = c == drop && i >= from;
                    const bool top = i % 3 == 2;
                    const float part = (float)(1 + c * 37 + t * 5 + i), v = top ? group_columns<RP, RP, true>(a, S, part, 0, c, seq)
                                                                               : group_columns<RP, RP, false>(a, S, part, 0, c, seq);
                    float want = 0.f;
                    for (int o = 0; o < C; ++o) want = top ? fmaxf(want, (float)(1 + o * 37 + t * 5 + i)) : want + (float)(1 + o * 37 + t * 5 + i);
                    if (v != want) { Hold h(mu); ++wrong; }
                    pthread_barrier_wait(&sync[c]);
                }
            });
    for (auto &t : all) t.join();
    printf("%d %d %d %d\n", wrong, status, g_armed_open, g_lost);
}
"""


def function(text, name):
    """A function of that name: its template line if it has one, up to the brace that closes it."""
    lines = text.split("\n")
    i = next(i for i, line in enumerate(lines) if line.startswith(("__device__", "__host__")) and f" {name}(" in line)
    first = i - 1 if lines[i - 1].startswith("template") else i
    last = i if lines[i].endswith("}") else lines.index("}", i)
    return "\n".join(lines[first:last + 1]) + "\n"


@pytest.fixture(scope="module")
def exchange(tmp_path_factory):
    text = open(CORE).read()
    d = tmp_path_factory.mktemp("exchange")
    (d / "x.cpp").write_text(FAKES + "".join(function(text, n) for n in ("wait_sends", "peer_bytes", "group_columns")) + MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-o", str(d / "x"), str(d / "x.cpp")], check=True)

    def run(*args):
        out = subprocess.run([str(d / "x")] + [str(a) for a in args], capture_output=True, text=True, check=True, timeout=300).stdout
        return dict(zip(("wrong", "status", "armed_open", "lost"), map(int, out.split())))
    return run


GROUPS = [(3, 3), (8, 8), (4, 2), (8, 4), (5, 1), (20, 1)]      # blocks, of a cluster


@pytest.mark.parametrize("C,K", GROUPS)
def test_totals(exchange, C, K):
    assert exchange(C, K, -1, 0) == dict(wrong=0, status=0, armed_open=0, lost=0)


@pytest.mark.parametrize("C,K", GROUPS)
def test_lost_messages_end_the_call_flagged(exchange, C, K):
    r = exchange(C, K, 1, 5)
    assert r["status"] == 4 and r["wrong"] > 0 and r["armed_open"] == 0
    # the exchange whose messages were lost and, in blocks of other clusters, the one after it; nothing is sent once a wait gave up
    assert r["lost"] <= 2 * 16 * (K + 1)
