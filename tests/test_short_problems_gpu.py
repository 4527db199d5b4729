"""Many short problems, one warp each (general path, r <= 32), against the float64 oracle: one row, rows at the edges of a warp's step (16
rows at r <= 16, 8 above), the largest that still takes the form, key lengths, token weights with a start, rebuilt kernels."""
import numpy as np
import pytest
import torch

from paper_2509_23436_b200 import synth
from lot_testutil import TOL, check_slice, gpu_forward, oracle_slices

pytestmark = pytest.mark.gpu
F32, BF16 = torch.float32, torch.bfloat16


# B, H, n, d, r, iters, eps, dtype, key mask, clustered
@pytest.mark.parametrize("case", [
    (60, 8, 1, 8, 5, 3, 0.1, F32, False, False),
    (60, 8, 15, 16, 16, 4, 0.1, BF16, False, False),
    (60, 8, 17, 24, 9, 4, 0.1, F32, True, False),
    (60, 8, 256, 16, 16, 3, 0.1, F32, False, False),
    (60, 8, 128, 32, 32, 5, 0.05, BF16, True, False),
    (60, 8, 9, 40, 17, 0, 0.1, F32, False, False),
    (60, 8, 100, 64, 30, 8, 0.01, F32, True, True),        # rebuilt, lost column sums
], ids=lambda c: "B%d-H%d-n%d-d%d-r%d-T%d-eps%g-%s%s%s" % (c[:7] + ("f32" if c[7] == F32 else "bf16", "-mask" if c[8] else "", "-peaked" if c[9] else "")))
def test_forward_matches_oracle(case):
    B, H, n, d, r, iters, eps, dtype, masked, peaked = case
    x = synth.make(B, H, n, d, r, seed=9600 + n + r, dtype=dtype, eps=eps, iters=iters,
                   key_len_range=(max(1, n // 2), n) if masked else None, qk="mixture" if peaked else "normal")
    res = gpu_forward(x, want_g=True)
    assert res["status"] == 0
    slices = [(0, 0), (B // 2, H // 2), (B - 1, H - 1)]
    outs, g1s, g2s = oracle_slices(x, slices, return_potentials=True)
    for (b, h), o, g1, g2 in zip(slices, outs, g1s, g2s):
        check_slice(res["out"][b, h], o, TOL[dtype], f"slice {(b, h)}")
        for got, ref in ((res["g1"][b, h], g1), (res["g2"][b, h], g2)):
            assert np.abs(got - ref).max() <= 1e-4 * max(1.0, np.abs(ref).max())
