"""Groups of more blocks than the sixteen words a thread waits for at once, exchanging through L2 (the long path), against the float64 oracle: a last turn
of words that is not full, key lengths that leave blocks without rows, kernels rebuilt and column sums redone on the way."""
import numpy as np
import pytest
import torch

from paper_2509_23436_b200 import binding as lot
from paper_2509_23436_b200 import synth
from lot_testutil import TOL, check_slice, gpu_forward, oracle_slices, to_dev
from test_launch_kind_gpu import launches

pytestmark = pytest.mark.gpu


# B, H, n, r, iters, eps, key lengths, clustered
@pytest.mark.parametrize("B,H,n,r,iters,eps,lens,peaked", [(1, 6, 20001, 64, 4, 0.1, None, False), (2, 3, 20000, 40, 3, 0.1, (30, 20000), False),
                                                           (1, 4, 65000, 64, 3, 0.1, None, False), (1, 6, 20000, 64, 5, 0.01, None, True)])
def test_forward_matches_oracle(B, H, n, r, iters, eps, lens, peaked):
    x = synth.make(B, H, n, 64, r, seed=60 + n, dtype=torch.bfloat16, eps=eps, iters=iters, key_len_range=lens, qk="mixture" if peaked else "normal")
    t = to_dev(x)
    args = [t[k] for k in ("q", "k", "v", "z", "beta", "key_len")]
    assert lot.lot_path(lot.LOT_BF16, B, H, n, 64, r, iters) == 4
    out, ws = lot.lot_attention_fwd_ex(*args, eps, iters)
    torch.cuda.synchronize()
    groups = [(blocks, cluster) for coop, cluster, blocks in launches(lambda: lot.lot_attention_fwd_ex(*args, eps, iters, out=out, ws=ws)) if coop]
    assert groups and groups[0][0] // (2 * B * H) // groups[0][1] > 16, groups
    res = gpu_forward(x, want_g=True)
    assert res["status"] == 0
    slices = sorted({(0, 0), (B - 1, H - 1)})
    outs, g1s, g2s = oracle_slices(x, slices, return_potentials=True)
    for (b, h), o, g1, g2 in zip(slices, outs, g1s, g2s):
        check_slice(res["out"][b, h], o, TOL[torch.bfloat16], f"slice {(b, h)}")
        # potentials of a bf16 kernel: 2e-4 of eps and more where few keys carry a column; the bound of the path's other tests
        for got, ref in ((res["g1"][b, h], g1), (res["g2"][b, h], g2)):
            assert np.abs(got - ref).max() <= 1e-3 * max(1.0, np.abs(ref).max())
    assert np.array_equal(res["out"], gpu_forward(x)["out"])
