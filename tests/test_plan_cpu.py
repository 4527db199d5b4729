"""How the general path splits a call over the device, by the library's own planning code compiled for the host: what a plan has to
promise whatever the sizes are.  Runs without a GPU (cluster limits are then the estimate the code falls back to)."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2509_23436_b200", "csrc")
SM_BYTES, RESERVE = 228 * 1024, 1024                       # shared memory of an SM, and what each block of it costs beyond its own

MAIN = r"""
#include "lot_sweep_plan.cu"
#include <cstdio>
namespace lot {
int device_sm_count() { return 148; }
namespace sweep {
cudaError_t launch_f32(const SweepPlan &, const SweepArgs &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_bf16(const SweepPlan &, const SweepArgs &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_keep(const SweepPlan &, const SweepArgs &, cudaStream_t) { return cudaSuccess; }
int cluster_count(int, size_t) { return 0; }
}
}
int main()
{
    int dt, BH, nq, nk, r, keep;
    while (scanf("%d %d %d %d %d %d", &dt, &BH, &nq, &nk, &r, &keep) == 6) {
        const lot::SweepPlan P = lot::sweep_plan(dt, BH, nq, nk, 64, r, keep != 0);
        printf("%d %d %d %d %d %d %d %d %d %zu\n", P.RP, P.C, P.K, P.groups, P.srows, P.tcols, P.threads, P.chained, ((nq > nk ? nq : nk) + P.C - 1) / P.C, P.smem);
    }
}
"""
FIELDS = ("RP", "C", "K", "groups", "srows", "tcols", "threads", "chained", "rows", "smem")


def sizes():
    """(dtype, slices, queries, keys, pivots, kept history), around the lines at which plans change and drawn ones."""
    some = [(0, 16, 700, 700, 64, 0), (0, 16, 1000, 1000, 32, 0), (1, 8, 500, 500, 64, 0), (1, 4, 2000, 2000, 16, 0), (0, 64, 200, 200, 64, 0), (1, 1, 1, 1, 256, 0),
            (1, 32, 16384, 16384, 256, 0), (0, 16, 16384, 16384, 64, 0), (1, 16, 4096, 4096, 64, 1), (0, 64, 333, 1531, 32, 0)]
    rng = random.Random(5)
    for _ in range(400):
        n = int(2 ** rng.uniform(0, 16))
        same = rng.random() < 0.7
        some.append((rng.randint(0, 1), int(2 ** rng.uniform(0, 9)), n, n if same else int(2 ** rng.uniform(0, 14)), rng.randint(1, 256), int(rng.random() < 0.3)))
    return some


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cu").write_text(MAIN)
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-cudart", "static", "-diag-suppress", "128",
                    "-I", CSRC, "-o", str(d / "plan"), str(d / "plan.cu")], check=True)
    asked = sizes()
    res = subprocess.run([str(d / "plan")], input="\n".join(" ".join(map(str, s)) for s in asked), capture_output=True, text=True, check=True)
    got = [dict(zip(FIELDS, map(int, line.split()))) for line in res.stdout.splitlines()]
    assert len(got) == len(asked)
    return list(zip(asked, got))


def test_a_block_with_tensor_memory_is_alone_on_its_sm(plans):
    """Two blocks of a group on one SM would wait for each other: one for the tensor memory, the other for its column sums.  Shared memory holds
    them apart whatever registers the compiler gives the kernel."""
    with_tensor = [(s, p) for s, p in plans if p["tcols"]]
    assert with_tensor
    for s, p in with_tensor:
        assert 2 * (p["smem"] + RESERVE) > SM_BYTES, (s, p)


def test_chained_clusters_leave_room(plans):
    """Clusters that start while their predecessor's last blocks run do not pack: a device's last ones would wait for the first to end.
    Cooperative groups are never chained, blocks on their own always."""
    for s, p in plans:
        blocks = p["groups"] * p["K"]
        if p["C"] == 1 or p["C"] > p["K"]:
            assert p["chained"] == (p["C"] == 1), (s, p)
        elif p["chained"]:
            slots = [148 * occ * 7 // 8 // p["K"] * p["K"] for occ in (1, 3)]              # what the planning code takes where no device answers
            alone = 2 * (p["smem"] + RESERVE) > SM_BYTES
            assert alone and blocks <= slots[0] and (p["K"] % 2 == 0 or 5 * blocks <= 4 * slots[0]) or not alone and 12 * blocks <= 11 * slots[1], (s, p)


def test_blocks_that_can_have_an_sm_each_do(plans):
    for s, p in plans:
        if p["threads"] > 32 and p["groups"] * p["C"] <= 148 * 7 // 8 // p["K"] * p["K"]:
            assert 2 * (p["smem"] + RESERVE) > SM_BYTES, (s, p)


def test_tensor_memory_is_taken_only_where_rows_go_there(plans):
    for s, p in plans:
        assert (p["tcols"] != 0) == (p["threads"] == 512 and p["rows"] > p["srows"]), (s, p)
