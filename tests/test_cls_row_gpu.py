"""The class token's softmax row where the blocks that share its keys can go wrong: one key, fewer keys than blocks, key counts that do
not divide, keys beyond what a block keeps in shared memory, key lengths that leave some blocks without keys."""
import numpy as np
import pytest
import torch

from paper_2509_23436_b200 import binding as lot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [(torch.float32, 1e-5), (torch.bfloat16, 5e-3)], ids=["f32", "bf16"])
@pytest.mark.parametrize("B,H,n,d,lens", [(1, 1, 2, 8, None), (2, 1, 257, 40, (3, 257)), (2, 6, 832, 64, (130, 832)), (1, 2, 1023, 256, None),
                                          (1, 1, 40001, 32, None), (2, 80, 300, 64, None)])
def test_softmax_row(B, H, n, d, lens, dtype, tol):
    """Against the plain softmax in float64: float32 sums, or the rounding of the output to bf16 (2^-9)."""
    g = torch.Generator().manual_seed(n + d)
    q, k, v = (torch.randn(B, H, n, d, generator=g).to(dtype) for _ in range(3))
    z, beta = torch.randn(H, 4, d, generator=g), torch.full((H, 4), 0.25)
    dev = torch.device("cuda:0")
    kl = None if lens is None else torch.tensor(lens, dtype=torch.int32, device=dev)
    tau = 0.7 * d ** -0.5
    out, ws = lot.lot_attention_fwd_var(q.to(dev), k.to(dev), v.to(dev), z.to(dev), beta.to(dev), 0.5, 1, key_len=kl, cls=True, cls_tau=tau)
    assert lot.lot_device_status(ws) in (0, 2)
    for b in range(B):
        m = n if lens is None else lens[b]
        w = torch.softmax(tau * (k[b, :, :m].double() @ q[b, :, 0].double().unsqueeze(-1)).squeeze(-1), dim=-1)
        ref = (w.unsqueeze(1) @ v[b, :, :m].double()).squeeze(1).numpy()
        got = out[b, :, 0].float().cpu().double().numpy()
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
