"""Two calls at once on two streams, each with its own workspace: the bits of the same calls one after the other, and no wait that runs out."""
import pytest
import torch

from paper_2509_23436_b200 import binding as lot
from paper_2509_23436_b200 import synth

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16
DEV = "cuda:0"

CALLS = {                                                       # B, H, n, d, r, dtype, backward
    "slice": (8, 3, 197, 64, 16, BF16, False),
    "general, a block a problem": (4, 12, 300, 32, 32, F32, False),
    "general, a cluster a problem": (1, 8, 900, 32, 128, BF16, False),
    "general, several clusters": (1, 1, 30001, 16, 64, F32, False),
    "long, a cluster a problem": (1, 16, 4096, 64, 64, BF16, False),
    "long, several clusters": (1, 2, 40000, 64, 64, BF16, False),
    "backward": (1, 4, 2000, 64, 64, BF16, True),
}
PAIRS = [("slice", "general, a cluster a problem"), ("general, a block a problem", "long, a cluster a problem"),
         ("general, a cluster a problem", "backward"), ("general, several clusters", "general, a cluster a problem"),
         ("long, several clusters", "slice"), ("general, several clusters", "long, several clusters")]


def prepared(name, seed):
    B, H, n, d, r, dtype, backward = CALLS[name]
    x = synth.make(B, H, n, d, r, seed=seed, dtype=dtype, eps=0.1, iters=5)
    t = [getattr(x, k).to(DEV) for k in ("q", "k", "v", "z", "beta")]
    if backward:
        dout = synth.cotangent(x).to(DEV)
        ws = lot.lot_attention_bwd(*t, None, dout, x.eps, x.iters)[5]
        return lambda: lot.lot_attention_bwd(*t, None, dout, x.eps, x.iters, ws=ws)[:5], ws
    out, ws = lot.lot_attention_fwd_ex(*t, None, x.eps, x.iters)
    return lambda: [lot.lot_attention_fwd_ex(*t, None, x.eps, x.iters, out=out, ws=ws)[0].clone()], ws


@pytest.mark.parametrize("pair", PAIRS, ids=lambda p: " and ".join(p).replace(", ", "-").replace(" ", "_"))
def test_calls_on_two_streams(pair):
    (one, ws1), (two, ws2) = prepared(pair[0], 1), prepared(pair[1], 2)
    want = one(), two()
    torch.cuda.synchronize()
    streams = torch.cuda.Stream(), torch.cuda.Stream()
    got = [], []
    for _ in range(6):
        for k, call in enumerate((one, two)):
            with torch.cuda.stream(streams[k]):
                got[k].append(call())
    torch.cuda.synchronize()
    assert lot.lot_device_status(ws1) == 0 and lot.lot_device_status(ws2) == 0
    for k in (0, 1):
        for res in got[k]:
            assert all(torch.equal(a, b) for a, b in zip(res, want[k]))
