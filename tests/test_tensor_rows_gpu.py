"""Groups of blocks that keep kernel rows in tensor memory and exchange their column sums through clusters, against the float64
oracle: a block alone, one cluster, several clusters of two and of four, the last row in shared memory, in tensor memory, in
its last step and behind it (streamed), token weights and key lengths over all of them, kernels rebuilt on the way, sides of
different lengths, and the reverse steps."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import lot_oracle as O
from oracle import lot_oracle_grad as OG
from paper_2509_23436_b200 import binding as lot
from paper_2509_23436_b200 import synth
from lot_testutil import TOL, check_slice, gpu_forward, oracle_slices
from test_backward_gpu import oracle_grads

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


def f64(t):
    return t.float().cpu().double().numpy()


# B, H, n, d, r, iters, eps, dtype, key mask, clustered
FORWARD = [
    (4, 50, 1500, 32, 64, 3, 0.1, BF16, False, False),     # alone, two steps of 64 rows in a lane's columns behind 768 rows
    (2, 35, 449, 32, 256, 3, 0.1, F32, True, False),       # alone, at the end of tensor memory (192 + 256 rows) and one row behind it
    (2, 35, 1000, 16, 200, 2, 0.1, BF16, False, False),    # ... many rows behind it
    (1, 8, 2000, 64, 256, 4, 0.1, BF16, True, False),      # a cluster of eight
    (3, 50, 2000, 32, 128, 3, 0.1, BF16, False, False),    # a cluster of three, problems in turns
    (1, 2, 6001, 32, 200, 3, 0.1, F32, True, False),       # clusters of two
    (1, 1, 16385, 32, 256, 3, 0.1, BF16, False, False),    # clusters of four
    (1, 1, 30001, 16, 32, 3, 0.1, F32, False, False),
    (1, 3, 9000, 128, 128, 6, 0.01, BF16, False, True),    # lost column sums, several rebuilds, across clusters
    (4, 50, 1500, 32, 64, 8, 0.01, BF16, True, True),      # ... in a block alone
]


@pytest.mark.parametrize("case", FORWARD, ids=lambda c: "B%d-H%d-n%d-d%d-r%d-T%d-eps%g-%s%s%s" % (
    c[:7] + ("f32" if c[7] == F32 else "bf16", "-mask" if c[8] else "", "-peaked" if c[9] else "")))
def test_forward_matches_oracle(case):
    B, H, n, d, r, iters, eps, dtype, masked, peaked = case
    x = synth.make(B, H, n, d, r, seed=9700 + n + r, dtype=dtype, eps=eps, iters=iters,
                   key_len_range=(max(1, n // 2), n) if masked else None, qk="mixture" if peaked else "normal")
    assert lot.lot_path(lot.LOT_F32 if dtype == F32 else lot.LOT_BF16, B, H, n, d, r, iters) == 0
    res = gpu_forward(x, want_g=True)
    assert res["status"] == 0
    slices = sorted({(0, 0), (B - 1, H - 1)})
    outs, g1s, g2s = oracle_slices(x, slices, return_potentials=True)
    for (b, h), o, g1, g2 in zip(slices, outs, g1s, g2s):
        check_slice(res["out"][b, h], o, TOL[dtype], f"slice {(b, h)}")
        for got, ref in ((res["g1"][b, h], g1), (res["g2"][b, h], g2)):
            assert np.abs(got - ref).max() <= 1e-4 * max(1.0, np.abs(ref).max())
    assert np.array_equal(res["out"], gpu_forward(x)["out"])


# B, H, nq, nk, r: the longer side first, its problems and the shorter one's shared by the same groups
@pytest.mark.parametrize("B,H,nq,nk,r", [(1, 2, 9000, 700, 33), (2, 30, 211, 2500, 64), (1, 1, 1, 20000, 16)])
def test_weighted_cross_attention_matches_oracle(B, H, nq, nk, r):
    d, eps, iters = 32, 0.1, 4
    rng = np.random.default_rng(5 + nq)
    q, k, v = (rng.standard_normal((B, H, m, d)).astype(np.float32) * d ** -0.5 for m in (nq, nk, nk))
    z = rng.standard_normal((H, r, d)).astype(np.float32)
    beta = rng.random((H, r)).astype(np.float32) + 0.2
    beta /= beta.sum(-1, keepdims=True)
    a, b = (rng.random((B, H, m)).astype(np.float32) + 0.1 for m in (nq, nk))
    a /= a.sum(-1, keepdims=True)
    b /= b.sum(-1, keepdims=True)
    dev = torch.device("cuda:0")
    t = [torch.from_numpy(x).to(dev) for x in (q, k, v, z, beta)]
    out = lot.lot_attention_fwd_var(*t, eps, iters, a=torch.from_numpy(a).to(dev), b=torch.from_numpy(b).to(dev))[0].cpu().numpy()
    for bb, h in {(0, 0), (B - 1, H - 1)}:
        ref = O.head_x(q[bb, h], k[bb, h], v[bb, h], z[h], beta[h], a[bb, h], b[bb, h], eps, iters)
        check_slice(out[bb, h], ref["out"], TOL[F32], f"slice {(bb, h)}")


# B, H, n, d, r, iters, eps, clustered
BACKWARD = [
    (4, 50, 1500, 32, 64, 3, 0.1, False),                  # alone
    (1, 8, 2000, 64, 256, 3, 0.1, False),                  # a cluster of eight
    (1, 2, 6001, 32, 200, 2, 0.1, False),                  # clusters of two
    (1, 2, 6000, 64, 128, 4, 0.02, True),                  # ... with rebuilt kernels
]


@pytest.mark.parametrize("case", BACKWARD, ids=lambda c: "B%d-H%d-n%d-d%d-r%d-T%d-eps%g%s" % (c[:7] + ("-peaked" if c[7] else "",)))
def test_backward_matches_oracle(case):
    B, H, n, d, r, iters, eps, peaked = case
    x = synth.make(B, H, n, d, r, seed=9800 + n + r, dtype=BF16, eps=eps, iters=iters, qk="mixture" if peaked else "normal")
    dout = synth.cotangent(x)
    dev = torch.device("cuda:0")
    t = [getattr(x, name).to(dev) for name in ("q", "k", "v", "z", "beta")]
    res = lot.lot_attention_bwd(*t, None, dout.to(dev), eps, iters)
    assert lot.lot_device_status(res[5]) == 0
    b, h = B - 1, H - 1                                        # the sums over slices are covered elsewhere
    one = dataclasses.replace(x, **{name: getattr(x, name)[b:, h:] for name in ("q", "k", "v")}, z=x.z[h:], beta=x.beta[h:])
    for name, got, ref in zip(("dq", "dk", "dv"), res, oracle_grads(one, dout[b:, h:])):
        check_slice(got[b, h].float().cpu().double().numpy(), ref[0, 0], TOL[BF16], name)


@pytest.mark.parametrize("B,H,n,d,r", [(1, 2, 6000, 32, 200), (4, 50, 1500, 32, 64), (60, 8, 60, 16, 16)])
def test_a_captured_call_gives_the_same_bits(B, H, n, d, r):
    """Cooperative launches in clusters, chained launches of blocks with tensor memory, one warp per problem."""
    x = synth.make(B, H, n, d, r, seed=3, dtype=F32 if d == 16 else BF16, eps=0.1, iters=3)
    dev = torch.device("cuda:0")
    t = [getattr(x, name).to(dev) for name in ("q", "k", "v", "z", "beta")]
    want, ws = lot.lot_attention_fwd_ex(*t, None, x.eps, x.iters)
    out = torch.zeros_like(want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        lot.lot_attention_fwd_ex(*t, None, x.eps, x.iters, out=out, ws=ws)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert lot.lot_device_status(ws) == 0 and torch.equal(out, want)


# H, n, r: padded ranks, rows in tensor memory and streamed ones
@pytest.mark.parametrize("H,n,r", [(200, 1500, 48), (200, 4000, 20)])
def test_backward_reversed_on_exponents_matches_oracle(H, n, r):
    """Potentials over more than the kept weights' range: such a problem's kernel is overwritten by exponents, -infinity in the padding."""
    d, eps, iters = 32, 0.01, 3
    x = synth.make(1, H, n, d, r, seed=9851 + n + r, dtype=BF16, eps=eps, iters=iters, qk="mixture")
    dout = synth.cotangent(x)
    f, w, h = x.f64(), np.full(n, 1.0 / n), H - 1
    fw = OG.head_forward(f["q"][0, h], f["k"][0, h], f["v"][0, h], f["z"][h], f["beta"][h], w, w, eps, iters)
    for trace, g in ((fw["tr1"], fw["g1"]), (fw["tr2"], fw["g2"])):
        all_g = np.array([g0 for g0, _ in trace] + [g]) / (eps * np.log(2))
        assert np.ptp(all_g, axis=0).max() > 230               # weights between 2^-115 and 2^115 cannot hold them
    dev = torch.device("cuda:0")
    t = [getattr(x, name).to(dev) for name in ("q", "k", "v", "z", "beta")]
    res = lot.lot_attention_bwd(*t, None, dout.to(dev), eps, iters)
    assert lot.lot_device_status(res[5]) == 0
    for name, got in zip(("dq", "dk", "dv", "dz", "dbeta"), res):
        assert bool(torch.isfinite(got.float()).all()), name
    ref = OG.head_backward(fw, f64(dout[0, h]))
    for name, got in zip(("dq", "dk", "dv"), res):
        check_slice(f64(got[0, h]), ref[name], TOL[BF16], name)
    check_slice(f64(res[3][h]), ref["dz"], TOL[BF16], "dz")
    check_slice(f64(res[4][h])[None, :], ref["dbeta"][None, :], TOL[BF16], "dbeta")
