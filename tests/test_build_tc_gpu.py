"""The Gibbs kernel built on tcgen05 (bf16 tokens, r > 32, d <= 128), through calls without iterations, whose plans are the row softmax
of the similarities: padded ranks and widths at their edges, rows at the edges of a tile, more tiles than blocks, heads beyond
the SMs, key lengths, skipped class token, starting potentials."""
import numpy as np
import pytest
import torch

from paper_2509_23436_b200 import binding as lot
from lot_testutil import TOL, check_slice

pytestmark = pytest.mark.gpu

# B, H, nq, nk, d, r, key lengths, starting potentials (query side, key side)
CASES = [
    (1, 1, 1, 2, 8, 33, None, (False, False)),
    (2, 3, 127, 129, 64, 64, None, (True, False)),
    (2, 2, 128, 257, 72, 65, (1, 200), (False, True)),
    (1, 2, 383, 640, 128, 128, None, (True, True)),
    (3, 2, 255, 130, 40, 129, (130, 64, 129), (False, False)),
    (2, 2, 500, 385, 128, 256, (385, 7), (False, True)),
    (1, 200, 60, 140, 16, 100, None, (False, False)),
    (6, 40, 300, 300, 24, 250, None, (False, False)),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "B%d-H%d-nq%d-nk%d-d%d-r%d%s" % (c[:6] + ("-mask" if c[6] else "",)))
def test_plans_without_iterations(case):
    B, H, nq, nk, d, r, lens, start = case
    g = torch.Generator().manual_seed(nq + nk + r)
    eps = 0.1
    q, k, v = ((torch.randn(B, H, n, d, generator=g) * d ** -0.5).to(torch.bfloat16) for n in (nq, nk, nk))
    z, beta = torch.randn(H, r, d, generator=g), torch.softmax(torch.randn(H, r, generator=g), -1)
    g1, g2 = (eps * torch.randn(B, H, r, generator=g) if s else None for s in start)
    dev = torch.device("cuda:0")
    up = lambda t: None if t is None else t.to(dev)
    kl = None if lens is None else torch.tensor(lens, dtype=torch.int32, device=dev)
    out, ws = lot.lot_attention_fwd_var(*(up(t) for t in (q, k, v, z, beta)), eps, 0, key_len=kl, g1_in=up(g1), g2_in=up(g2))
    assert lot.lot_device_status(ws) == 0
    got = out.float().cpu().double().numpy()
    for b, h in {(0, 0), (B - 1, H - 1), (B // 2, H // 2)}:
        m = nk if lens is None else lens[b]

        def plan(x, gg):
            s = x.double() @ z[h].double().T
            return torch.softmax((s + (0 if gg is None else gg[b, h].double())) / eps, -1)
        w = plan(k[b, h, :m], g2).T @ v[b, h, :m].double() / m / beta[h].double().unsqueeze(-1)
        check_slice(got[b, h], (plan(q[b, h], g1) @ w).numpy(), TOL[torch.bfloat16], f"slice {(b, h)}")


def test_class_token_is_skipped():
    B, H, n, d, r = 1, 2, 258, 64, 64
    g = torch.Generator().manual_seed(3)
    q, k, v = ((torch.randn(B, H, n, d, generator=g) * d ** -0.5).to(torch.bfloat16) for _ in range(3))
    z, beta = torch.randn(H, r, d, generator=g), torch.full((H, r), 1.0 / r)
    dev = torch.device("cuda:0")
    t = [x.to(dev) for x in (q, k, v, z, beta)]
    whole = lot.lot_attention_fwd_var(*t, 0.1, 3, cls=True)[0][:, :, 1:].float().cpu().numpy()
    part = lot.lot_attention_fwd_var(*(x[:, :, 1:].contiguous() for x in t[:3]), t[3], t[4], 0.1, 3)[0].float().cpu().numpy()
    assert np.abs(whole - part).max() <= 2.0 ** -8 * np.abs(part).max()          # two roundings to bf16
