"""What the sizes around the long path keep of float32: the key side of the read-out, the first pivot updates, the iterations at
r <= 32, and calls whose output lies over an input."""
import numpy as np
import pytest
import torch

from paper_2509_23436_b200 import binding as lot
from paper_2509_23436_b200 import synth
from lot_testutil import check_slice, gpu_forward, oracle_slices, to_dev

pytestmark = pytest.mark.gpu
BF16, LONG = torch.bfloat16, 4


@pytest.mark.parametrize("n, masked", [(4096, False), (4001, True), (16384, False)])
def test_key_side_is_applied_from_more_than_bf16(n, masked):
    """Every query sits on one pivot (all others 2^-170 below), and as many on each: out_i is a row of W', whose error is the
    key side's.  A bf16 plan would add noise of 2^-9 / sqrt(3) = 1.1e-3 of the rms, up to four times that among 8192
    entries; what is left is the output's own rounding (half a unit in the last place, at most 2^-8 of the entry) and
    the potentials' error (1.6e-4 at this eps, doubled by the row sums)."""
    x = synth.make(1, 2, n, 64, 64, seed=77 + n, dtype=BF16, eps=0.1, iters=10, key_len_range=(n // 2, n) if masked else None)
    x.z.copy_(torch.eye(64).expand(2, 64, 64))
    x.beta.fill_(1 / 64)
    x.q.zero_()
    x.q[:, :, torch.arange(n), torch.arange(n) % 64] = 12.
    x.k.copy_((x.k.float() / x.k.float().norm(dim=3, keepdim=True)).to(BF16))
    assert lot.lot_path(lot.LOT_BF16, 1, 2, n, 64, 64, 10) == LONG
    res = gpu_forward(x)
    assert res["status"] == 0
    for h, ref in enumerate(oracle_slices(x, [(0, 0), (0, 1)])):
        excess = np.abs(res["out"][0, h] - ref) - 2 ** -8 * np.abs(ref)
        assert excess.max() <= 5e-4 * np.sqrt((ref ** 2).mean())


def split_pivot_bound(x):
    """What pivots as bf16 hi + lo leave of the logits' accuracy, in units of the potentials: 2^-18 of every product of a token
    with a pivot, d errors of either sign, taken twice.  The iterations on float32 values add 1e-6; a bf16 kernel moves the
    potentials by one and a half to nine times this bound at the sizes below."""
    q, z = x.q.float().norm(dim=3).pow(2).mean().sqrt(), x.z.norm(dim=2).max()
    return 2 * 2 ** -18 * float(q * z) / np.sqrt(x.shape[3])


# one update; ten at r <= 32 on both sides of the line between the general and the streamed path
@pytest.mark.parametrize("shape, iters", [((1, 2, 4096, 64, 64), 1), ((4, 3, 700, 64, 40), 1), ((1, 64, 2048, 64, 32), 10),
                                          ((1, 12, 12000, 64, 24), 10), ((1, 16, 12288, 64, 32), 10)])
def test_iterations_are_on_float32_values(shape, iters):
    x = synth.make(*shape, seed=55, dtype=BF16, eps=0.1, iters=iters)
    res = gpu_forward(x, want_g=True)
    assert res["status"] == 0
    slices = [(0, 0), (0, shape[1] - 1)]
    for (b, h), o, g1, g2 in zip(slices, *oracle_slices(x, slices, return_potentials=True)):
        check_slice(res["out"][b, h], o, 2e-2)
        for got, ref in ((res["g1"][b, h], g1), (res["g2"][b, h], g2)):
            assert np.abs(got - ref).max() <= split_pivot_bound(x)


@pytest.mark.parametrize("over", ["q", "k", "v"])
def test_output_over_an_input(over):
    x = synth.make(1, 3, 2500, 64, 50, seed=91, dtype=BF16, eps=0.1, iters=6)
    ref = oracle_slices(x, [(0, 0), (0, 2)])
    t = to_dev(x)
    out, ws = lot.lot_attention_fwd_ex(t["q"], t["k"], t["v"], t["z"], t["beta"], None, x.eps, x.iters, out=t[over])
    torch.cuda.synchronize()
    assert lot.lot_device_status(ws) == 0
    got = out.float().cpu().double().numpy()
    for h, r in zip((0, 2), ref):
        check_slice(got[0, h], r, 2e-2)
