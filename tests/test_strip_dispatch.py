"""Which sides above 32 take the register tiles, on the CPU: windows that fill little of their 32-slot strips and 128-slot tiles, told by the
workspace that the calls ask for (the register tiles': none forward, a float per token and head backward)."""
import pytest

import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import small_config

CASES = [
    # B, H, W, heads, head_dim, window -> strips forward, backward
    ((1, 240, 360, 6, 32, 33), False, True), ((1, 240, 360, 6, 32, 38), False, True), ((1, 240, 360, 6, 32, 40), True, True), ((1, 96, 180, 6, 64, 33), True, True),
    ((1, 96, 180, 4, 128, 33), True, True), ((200, 64, 1, 6, 32, 64), False, False), ((8, 128, 4, 12, 128, 64), False, False), ((200, 8, 8, 4, 128, 40), False, False),
    ((1, 8, 8, 2, 64, 128), False, False), ((1, 10, 32, 2, 32, 64), False, True), ((1, 12, 32, 2, 32, 64), True, True), ((1, 8, 32, 2, 64, 64), False, True),
    ((1, 4, 32, 2, 128, 64), False, True), ((1, 8, 32, 2, 128, 64), True, True), ((1, 256, 640, 8, 128, 128), True, True), ((1, 64, 64, 1, 32, 64), True, True),
]


@pytest.mark.parametrize("case, forward, backward", CASES, ids=["_".join(map(str, c[0])) for c in CASES])
def test_route(case, forward, backward):
    B, H, W, heads, head_dim, window = case
    for dtype in (0, 1):
        desc = terra.make_desc(small_config("route", B, H, W, heads, head_dim, window, 0, window // 2))
        desc.dtype = dtype
        delta = -(-4 * B * H * W * heads // 256) * 256
        assert (terra.terra_swin_workspace_bytes(desc, False) > 0) == forward
        assert (terra.terra_swin_workspace_bytes(desc, True) > delta) == backward


OWN = [
    # B, H, W, heads, head_dim, window, shift_h, shift_w, periodic_h, periodic_w: complete windows of side 64 and 128 on their own forward kernel or not
    ((1, 64, 640, 1, 64, 64, 0, 8, 0, 1), True), ((1, 64, 576, 1, 64, 64, 0, 8, 0, 1), False), ((1, 128, 256, 16, 128, 128, 64, 64, 1, 1), True),
    ((1, 128, 256, 16, 128, 128, 64, 64, 0, 1), False), ((1, 128, 256, 16, 128, 128, 0, 64, 0, 0), False), ((1, 128, 256, 16, 128, 128, 0, 60, 0, 1), False),
    ((1, 64, 64, 40, 64, 64, 0, 0, 0, 1), False), ((1, 64, 64, 37, 64, 64, 0, 0, 0, 1), True), ((1, 64, 64, 149, 64, 64, 0, 0, 0, 1), False),
    ((1, 128, 256, 16, 32, 128, 0, 64, 0, 1), False), ((1, 128, 320, 16, 128, 96, 0, 64, 0, 1), False),
]


@pytest.mark.parametrize("case, own", OWN, ids=["_".join(map(str, c[0])) for c in OWN])
def test_complete_windows_route(case, own):
    desc = terra.make_desc(small_config("route", *case))
    heads, window = case[3], case[5]
    prepared = -(-4 * heads * ((2 * window - 1) * 2 * window + 4) // 256) * 256          # that kernel's tables; strips' are larger
    assert (terra.terra_swin_workspace_bytes(desc, False) == prepared) == own
