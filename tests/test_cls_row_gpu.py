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


@pytest.mark.parametrize("bad", [float("nan"), float("-inf"), float("inf")], ids=["nan", "neg_inf", "inf"])
@pytest.mark.parametrize("n,length,which", [(257, 3, (0,)), (257, 3, (2,)), (257, 3, (1, 2)), (257, 3, (0, 1, 2)), (832, 832, (831,)), (832, 832, range(140)),
                                            (100, 100, (50,))])
def test_keys_that_score_no_number(n, length, which, bad):
    """A key that scores NaN makes the row NaN and one of -infinity weighs nothing, whichever share it is in and whether or not it
    is alone there: as the softmax in float64 has it."""
    d = 16
    g = torch.Generator().manual_seed(n)
    q, k, v = (torch.randn(1, 1, n, d, generator=g) for _ in range(3))
    q[0, 0, 0] = q[0, 0, 0].abs() + 0.1                             # so that the score has the entry's sign
    for j in which:
        k[0, 0, j, 3] = bad
    z, beta = torch.randn(1, 4, d, generator=g), torch.full((1, 4), 0.25)
    dev = torch.device("cuda:0")
    out, _ = lot.lot_attention_fwd_var(q.to(dev), k.to(dev), v.to(dev), z.to(dev), beta.to(dev), 0.5, 1,
                                       key_len=torch.tensor([length], dtype=torch.int32, device=dev), cls=True, cls_tau=0.2)
    ref = torch.softmax(0.2 * (k[0, 0, :length].double() @ q[0, 0, 0].double()), dim=-1) @ v[0, 0, :length].double()
    got = out[0, 0, 0].double().cpu()
    assert torch.equal(torch.isnan(got), torch.isnan(ref))
    if not torch.isnan(ref).any():
        assert (got - ref).abs().max() <= 1e-5 * ref.abs().max()
