"""The general path's sweep kernels (scaling form on a stored float32 Gibbs kernel) against the float64 oracle where they can
go wrong: padded ranks at both sides of 16, 32, 64, 128, 256; rows at the edges of row tiles and steps; one block per
problem, groups that exchange every word and groups with per-column owners; rows that do not fit shared memory; one
launch per pass; potentials that leave the kernel's range (rebuilding, lost column sums) forward and backward."""
import numpy as np
import pytest
import torch

from paper_2509_23436_b200 import binding as lot
from paper_2509_23436_b200 import synth
from lot_testutil import TOL, check_slice, gpu_forward, oracle_slices
from test_backward_gpu import oracle_grads

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16

# B, H, n, d, r, iters, eps, dtype, key mask, clustered
FORWARD = [
    (1, 1, 1, 8, 1, 3, 0.1, F32, False, False),
    (1, 2, 127, 24, 16, 4, 0.1, F32, True, False),
    (1, 2, 129, 72, 17, 4, 0.1, BF16, False, False),
    (2, 2, 513, 32, 32, 0, 0.1, F32, False, False),        # no iteration
    (1, 2, 1025, 128, 33, 3, 0.1, BF16, True, False),
    (1, 3, 2049, 64, 65, 3, 0.1, BF16, False, False),
    (1, 1, 4097, 256, 129, 2, 0.1, F32, False, False),     # widest tokens, row tiles of eight
    (1, 2, 600, 256, 30, 3, 0.1, BF16, False, False),
    (1, 2, 3001, 128, 256, 3, 0.1, BF16, True, False),     # group with per-column owners
    (200, 2, 80, 64, 8, 5, 0.1, F32, True, False),         # more problems than blocks
    (1, 1, 70001, 64, 64, 2, 0.1, F32, False, False),      # rows streamed
    (1, 4, 70001, 64, 64, 2, 0.1, F32, False, False),      # one launch per pass
    (1, 2, 1200, 128, 64, 20, 0.01, BF16, False, True),    # lost column sums, several rebuilds
    (1, 2, 700, 128, 256, 8, 0.01, F32, True, True),
    (1, 1, 9000, 128, 128, 6, 0.02, BF16, False, True),    # the same across a group
    (1, 2, 300, 64, 12, 50, 0.02, F32, False, True),
]


@pytest.mark.parametrize("case", FORWARD, ids=lambda c: "B%d-H%d-n%d-d%d-r%d-T%d-eps%g-%s%s%s" % (
    c[:7] + ("f32" if c[7] == F32 else "bf16", "-mask" if c[8] else "", "-peaked" if c[9] else "")))
def test_forward_matches_oracle(case):
    B, H, n, d, r, iters, eps, dtype, masked, peaked = case
    x = synth.make(B, H, n, d, r, seed=9000 + n + r, dtype=dtype, eps=eps, iters=iters,
                   key_len_range=(max(1, n // 2), n) if masked else None, qk="mixture" if peaked else "normal")
    assert lot.lot_path(lot.LOT_F32 if dtype == F32 else lot.LOT_BF16, B, H, n, d, r, iters) == 0
    res = gpu_forward(x, want_g=True)
    assert res["status"] == 0
    slices = sorted({(0, 0), (B // 2, H // 2), (B - 1, H - 1)})
    outs, g1s, g2s = oracle_slices(x, slices, return_potentials=True)
    for (b, h), o, g1, g2 in zip(slices, outs, g1s, g2s):
        check_slice(res["out"][b, h], o, TOL[dtype], f"slice {(b, h)}")
        for got, ref in ((res["g1"][b, h], g1), (res["g2"][b, h], g2)):
            assert np.abs(got - ref).max() <= 1e-4 * max(1.0, np.abs(ref).max())
    again = gpu_forward(x)
    assert np.array_equal(res["out"], again["out"])


# bf16 tensors run on the stored kernel in reverse too
BACKWARD = [
    (1, 1, 2, 16, 3, 2, 0.1, False, False),
    (2, 3, 127, 64, 16, 10, 0.1, True, False),
    (1, 2, 257, 40, 33, 4, 0.1, False, False),
    (1, 2, 1030, 128, 65, 3, 0.1, True, False),
    (1, 1, 1500, 128, 256, 3, 0.1, False, False),
    (1, 1, 3000, 256, 20, 0, 0.1, False, False),
    (1, 2, 600, 128, 64, 6, 0.05, False, True),            # rebuilt kernel, kept weights still in range
    (1, 2, 500, 128, 32, 6, 0.01, True, True),             # ... out of range: step by step
]


@pytest.mark.parametrize("case", BACKWARD, ids=lambda c: "B%d-H%d-n%d-d%d-r%d-T%d-eps%g%s%s" % (
    c[:7] + ("-mask" if c[7] else "", "-peaked" if c[8] else "")))
def test_backward_matches_oracle(case):
    B, H, n, d, r, iters, eps, masked, peaked = case
    x = synth.make(B, H, n, d, r, seed=9500 + n + r, dtype=BF16, eps=eps, iters=iters,
                   key_len_range=(max(1, n // 2), n) if masked else None, qk="mixture" if peaked else "normal")
    dout = synth.cotangent(x)
    dev = torch.device("cuda:0")
    kl = None if x.key_len is None else x.key_len.to(dev)
    t = [getattr(x, name).to(dev) for name in ("q", "k", "v", "z", "beta")]
    runs = []
    for _ in range(2):
        res = lot.lot_attention_bwd(*t, kl, dout.to(dev), eps, iters)
        torch.cuda.synchronize()
        assert lot.lot_device_status(res[5]) == 0
        runs.append([g.float().cpu().double().numpy() for g in res[:5]])
    ref = oracle_grads(x, dout)
    for i, name in enumerate(("dq", "dk", "dv")):
        for b in range(B):
            for h in range(H):
                check_slice(runs[0][i][b, h], ref[i][b, h], 2e-2, f"{name} {(b, h)}")
    for i, name in ((3, "dz"), (4, "dbeta")):
        for h in range(H):
            check_slice(runs[0][i][h], ref[i][h], 2e-2, f"{name} head {h}")
    for a, b in zip(*runs):
        assert np.array_equal(a, b)


# the long path: bf16 kernel, d = 64, 16 < r <= 64 (the library's own choice from three iterations on); B, H, n, r, iters, eps, key mask, clustered
LONG = [
    (1, 2, 1, 33, 2, 0.1, False, False),
    (1, 2, 127, 40, 5, 0.1, True, False),
    (1, 1, 1000, 64, 0, 0.1, False, False),
    (2, 3, 1153, 33, 4, 0.05, True, False),
    (2, 3, 1153, 17, 4, 0.05, True, False),
    (1, 2, 2048, 32, 6, 0.1, False, False),
    (1, 1, 20000, 64, 4, 0.1, False, False),               # rows streamed
    (40, 8, 300, 64, 3, 0.1, True, False),                 # one block per problem
    (1, 3, 65536, 50, 2, 0.1, False, False),
    (1, 2, 3000, 64, 8, 0.02, False, True),                # rebuilt kernel
    (1, 1, 1500, 50, 12, 0.01, True, True),                # lost column sums, final potentials far apart
    (1, 2, 1000, 50, 12, 0.01, True, True),                # the same in a cluster of eight blocks
    (3, 16, 1024, 64, 5, 0.05, True, False),
]


@pytest.mark.parametrize("case", LONG, ids=lambda c: "B%d-H%d-n%d-r%d-T%d-eps%g%s%s" % (
    c[:6] + ("-mask" if c[6] else "", "-peaked" if c[7] else "")))
def test_long_path_matches_oracle(case):
    B, H, n, r, iters, eps, masked, peaked = case
    x = synth.make(B, H, n, 64, r, seed=9800 + n + r, dtype=BF16, eps=eps, iters=iters,
                   key_len_range=(max(1, n // 2), n) if masked else None, qk="mixture" if peaked else "normal")
    lot.lot_debug_hook(4, 4)
    try:
        assert lot.lot_path(lot.LOT_BF16, B, H, n, 64, r, iters) == 4
        res, again = gpu_forward(x, want_g=True), gpu_forward(x)
    finally:
        lot.lot_debug_hook(4, -1)
    assert res["status"] == 0 and np.array_equal(res["out"], again["out"])
    slices = sorted({(0, 0), (B // 2, H // 2), (B - 1, H - 1)})
    outs, g1s, g2s = oracle_slices(x, slices, return_potentials=True)
    for (b, h), o, g1, g2 in zip(slices, outs, g1s, g2s):
        check_slice(res["out"][b, h], o, 2e-2, f"slice {(b, h)}")
        for got, ref in ((res["g1"][b, h], g1), (res["g2"][b, h], g2)):
            assert np.abs(got - ref).max() <= 1e-3 * max(1.0, np.abs(ref).max())
