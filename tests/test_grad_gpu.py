"""The last stage of the backward of bf16 tensors (gradients of similarities put together and multiplied in one kernel) against the
oracle's gradients: every kernel shape, rows at the edges of a step of 64 and of a chunk, iterations at the edges of what is
staged together (8, 16), no iteration, key lengths down to two keys, and a batch row without any."""
import pytest
import torch

import numpy as np
from paper_2509_23436_b200 import binding as lot
from paper_2509_23436_b200 import synth
from lot_testutil import check_slice
from test_backward_gpu import oracle_grads

pytestmark = pytest.mark.gpu

# B, H, n, d, r, iters, key lengths
CASES = [
    (1, 1, 2, 8, 3, 1, None),                              # one token or one key: gradients of exactly zero, nothing to compare with
    (1, 2, 63, 64, 16, 16, None),
    (2, 1, 64, 40, 9, 17, (2, 64)),
    (2, 1, 65, 128, 16, 0, (65, 33)),
    (1, 2, 257, 64, 32, 33, None),
    (2, 1, 321, 72, 17, 5, (64, 257)),
    (1, 2, 513, 64, 64, 15, None),
    (2, 2, 300, 128, 64, 8, (129, 300)),
    (1, 1, 400, 120, 33, 9, None),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d-H%d-n%d-d%d-r%d-T%d%s" % (c[:6] + ("-mask" if c[6] else "",)))
def test_gradients_match_oracle(case):
    B, H, n, d, r, iters, lens = case
    x = synth.make(B, H, n, d, r, seed=9900 + n + r, dtype=torch.bfloat16, eps=0.1, iters=iters)
    if lens:
        x.key_len = torch.tensor(lens, dtype=torch.int32)
    dout = synth.cotangent(x)
    dev = torch.device("cuda:0")
    t = [getattr(x, name).to(dev) for name in ("q", "k", "v", "z", "beta")]
    res = lot.lot_attention_bwd(*t, None if not lens else x.key_len.to(dev), dout.to(dev), x.eps, iters)
    assert lot.lot_device_status(res[5]) == 0
    got = [g.float().cpu().double().numpy() for g in res[:5]]
    ref = oracle_grads(x, dout)
    for i, name in enumerate(("dq", "dk", "dv")):
        for b in range(B):
            for h in range(H):
                check_slice(got[i][b, h], ref[i][b, h], 2e-2, f"{name} {(b, h)}")
    for i, name in ((3, "dz"), (4, "dbeta")):
        for h in range(H):
            check_slice(got[i][h], ref[i][h], 2e-2, f"{name} head {h}")


def test_a_batch_row_without_keys_has_finite_gradients():
    x = synth.make(2, 2, 130, 64, 32, seed=9999, dtype=torch.bfloat16, eps=0.1, iters=4)
    dev = torch.device("cuda:0")
    t = [getattr(x, name).to(dev) for name in ("q", "k", "v", "z", "beta")]
    ws = torch.full((lot.lot_bwd_workspace_bytes(2, 2, 130, 64, 32, lot.LOT_BF16, 4),), 0xFF, dtype=torch.uint8, device=dev)
    res = lot.lot_attention_bwd(*t, torch.tensor([0, 130], dtype=torch.int32, device=dev), synth.cotangent(x).to(dev), 0.1, 4, ws=ws)
    assert np.all(res[1][0].float().cpu().numpy() == 0) and np.all(res[2][0].float().cpu().numpy() == 0)
    for g in res[:5]:
        assert bool(torch.isfinite(g.float()).all())
    assert np.all(res[0][0].float().cpu().numpy() == 0)
    # the sums over the batch are the other row's: float32 sums of at most 130 tokens in another order, through four reverse steps
    one = lot.lot_attention_bwd(*(g[1:].contiguous() for g in t[:3]), *t[3:], None, synth.cotangent(x)[1:].contiguous().to(dev), 0.1, 4)
    for i, name in ((3, "dz"), (4, "dbeta")):
        for h in range(2):
            check_slice(res[i][h].cpu().double().numpy(), one[i][h].cpu().double().numpy(), 1e-4, f"{name} head {h}")
