"""Calls on the stored kernel whose workspace would pass 8 GiB run their slices in parts: the same bits as separate calls of
the parts, dz and dbeta their sum over the batch."""
import pytest
import torch

from paper_2509_23436_b200 import binding as lot

pytestmark = pytest.mark.gpu
N, D, R, EPS, T = 4096, 8, 16, 0.1, 10
LIMIT = 8 << 30


def draw(B, H, count):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(B * 1000 + H)
    x = [torch.randn(B, H, N, D, generator=gen, device="cuda", dtype=torch.bfloat16).mul_(D ** -0.5) for _ in range(count)]
    z = torch.randn(H, R, D, generator=gen, device="cuda")
    beta = torch.softmax(torch.randn(H, R, generator=gen, device="cuda"), 1).contiguous()
    key_len = torch.randint(N // 2, N + 1, (B,), generator=gen, device="cuda", dtype=torch.int32)
    key_len[0] = 0                                          # its flag is raised in the first part and must outlive the others
    return x, z, beta, key_len


# rows of the batch in two parts; heads of each row in two
@pytest.mark.parametrize("B, H, rows, heads", [(64, 128, 32, 128), (2, 8192, 1, 4096)])
def test_backward_in_parts(B, H, rows, heads):
    (q, k, v, dout), z, beta, key_len = draw(B, H, 4)
    assert lot.lot_bwd_workspace_bytes(B, H, N, D, R, lot.LOT_BF16, T) <= LIMIT
    *whole, ws = lot.lot_attention_bwd(q, k, v, z, beta, key_len, dout, EPS, T)
    assert lot.lot_device_status(ws) == lot.LOT_DEV_EMPTY
    dz, dbeta = torch.zeros_like(z), torch.zeros_like(beta)
    for b in range(0, B, rows):
        for h in range(0, H, heads):
            part = lambda t: t[b:b + rows, h:h + heads].contiguous()
            *res, _ = lot.lot_attention_bwd(part(q), part(k), part(v), z[h:h + heads].contiguous(), beta[h:h + heads].contiguous(),
                                            key_len[b:b + rows].clone(), part(dout), EPS, T, ws=ws)
            for a, g in zip(whole, res[:3]):
                assert torch.equal(part(a), g)
            dz[h:h + heads] += res[3]
            dbeta[h:h + heads] += res[4]
    assert torch.equal(whole[3], dz) and torch.equal(whole[4], dbeta)


def test_forward_in_parts():
    B, H = 128, 128
    (q, k, v), z, beta, key_len = draw(B, H, 3)
    assert lot.lot_workspace_bytes(B, H, N, D, R, lot.LOT_BF16) <= LIMIT
    g1, g2 = (torch.empty(B, H, R, device="cuda") for _ in range(2))
    out, ws = lot.lot_attention_fwd_ex(q, k, v, z, beta, key_len, EPS, T, g1_out=g1, g2_out=g2)
    assert lot.lot_device_status(ws) == lot.LOT_DEV_EMPTY
    for b in (0, 64):
        s = slice(b, b + 64)
        h1, h2 = torch.empty_like(g1[s]), torch.empty_like(g2[s])
        part, _ = lot.lot_attention_fwd_ex(q[s], k[s], v[s], z, beta, key_len[s].clone(), EPS, T, g1_out=h1, g2_out=h2, ws=ws)
        assert torch.equal(out[s], part) and torch.equal(g1[s][1:], h1[1:]) and torch.equal(g2[s][1:], h2[1:])
