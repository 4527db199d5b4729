"""Which path a call takes and the workspace it asks for, where the rule has a line (host arithmetic, no GPU; 148 SMs)."""
import pytest

from paper_2509_23436_b200 import binding as lot
from paper_2509_23436_b200 import build as lot_build

GENERAL, STREAMED, SLICE, LONG = 0, 1, 3, 4

# B, H, n, r, iters, path
LINES = [
    (1, 16, 16384, 64, 10, LONG), (1, 16, 16384, 64, 3, LONG), (1, 16, 16384, 64, 2, STREAMED), (1, 16, 16384, 64, 0, STREAMED),
    (1, 16, 18750, 33, 10, LONG), (1, 16, 18751, 33, 10, STREAMED), (32, 16, 1200, 64, 10, LONG), (32, 16, 1201, 64, 10, STREAMED),
    (1, 16, 6250, 32, 10, GENERAL), (1, 16, 10000, 32, 10, GENERAL), (1, 16, 10001, 32, 10, STREAMED), (1, 600, 1200, 32, 10, GENERAL),
    # r <= 32 on a bf16 kernel only at about one slice of up to 14 tiles per SM
    (1, 74, 1400, 32, 10, LONG), (1, 73, 1400, 32, 10, GENERAL), (1, 148, 1792, 17, 3, LONG), (1, 148, 1792, 17, 2, STREAMED),
    (1, 149, 1792, 32, 10, STREAMED), (1, 148, 1793, 32, 10, STREAMED), (1, 148, 1200, 32, 10, GENERAL),
    (1, 16, 65536, 16, 10, GENERAL), (32, 3, 197, 16, 10, SLICE),
]


@pytest.fixture(scope="module")
def L():
    lot_build.build_lib()
    return lot.lib()


@pytest.mark.parametrize("case", LINES, ids=lambda c: "B%d-H%d-n%d-r%d-T%d" % c[:5])
def test_path(L, case):
    B, H, n, r, iters, path = case
    assert L.lot_path(lot.LOT_BF16, B, H, n, 64, r, iters) == path


def test_workspace_serves_any_number_of_iterations(L):
    """The size does not depend on the iterations, so it is that of the path that needs most."""
    for B, H, n, r, _, _ in LINES:
        size = L.lot_workspace_bytes(B, H, n, 64, r, lot.LOT_BF16)
        for path in {L.lot_path(lot.LOT_BF16, B, H, n, 64, r, t) for t in (0, 1, 2, 3, 50)}:
            if path in (STREAMED, LONG):
                assert L.lot_debug_hook(4, path) == 0
                try:
                    assert size >= L.lot_workspace_bytes(B, H, n, 64, r, lot.LOT_BF16)
                finally:
                    L.lot_debug_hook(4, -1)


def test_empty_problems_have_a_path(L):
    for B, n in ((0, 1000), (2, 0), (0, 0)):
        assert L.lot_path(lot.LOT_BF16, B, 4, n, 64, 64, 10) == GENERAL
        assert L.lot_workspace_bytes(B, 4, n, 64, 64, lot.LOT_BF16) > 0


def test_workspace_of_large_calls_is_bounded(L):
    """Slices beyond 8 GiB of workspace go in parts; a slice by itself is never split, and float32 tensors keep the size they
    always asked for."""
    limit = 8 << 30
    assert L.lot_bwd_workspace_bytes(64, 128, 4096, 8, 16, lot.LOT_BF16, 10) <= limit
    assert L.lot_bwd_workspace_bytes(2, 8192, 4096, 8, 16, lot.LOT_BF16, 50) <= limit
    assert L.lot_bwd_workspace_bytes(1, 7, 1 << 22, 64, 256, lot.LOT_BF16, 50) == L.lot_bwd_workspace_bytes(1, 1, 1 << 22, 64, 256, lot.LOT_BF16, 50) > limit
    assert L.lot_workspace_bytes(512, 64, 8000, 32, 129, lot.LOT_BF16) <= limit
    assert L.lot_var_workspace_bytes(512, 63, 8000, 777, 32, 129, lot.LOT_BF16) <= limit
    assert L.lot_workspace_bytes(512, 63, 8000, 32, 129, lot.LOT_F32) >= 512 * 63 * 16000 * 129 * 8
    assert L.lot_launch_count(lot.LOT_BF16, 128, 128, 4096, 8, 16, 10) == 8 and L.lot_launch_count(lot.LOT_BF16, 12, 128, 4096, 8, 16, 10) == 4
    # below the limit it is that of one part
    one = L.lot_bwd_workspace_bytes(1, 16, 4096, 64, 64, lot.LOT_BF16, 10)
    assert one < 3 * 2 * 16 * 4096 * 64 * 4
