"""The forward kernel for window sides 9 .. 32 at the edges of its range: both slot layouts, one and two query tiles, an odd number of
them, half a chunk of keys and less, truncated windows, seams that cut a window column at an odd token, runs of units that change
their head, and bias tables that raise the softmax reference in the middle of a row.  Against the oracle."""
import pytest
import torch

import oracle
import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config
from tests._parity import gate, gpu_rows

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, W, heads, head_dim, window, shift_h, shift_w, periodic_h, periodic_w
    (2, 27, 30, 2, 64, 9, 4, 3, 0, 1), (1, 41, 50, 2, 128, 13, 6, 5, 0, 0), (1, 48, 80, 3, 128, 16, 0, 0, 0, 1), (2, 80, 70, 5, 64, 17, 8, 9, 1, 0),
    (2, 45, 50, 2, 64, 20, 10, 10, 0, 1), (1, 70, 45, 2, 64, 31, 20, 30, 0, 0), (1, 60, 73, 3, 32, 24, 12, 12, 0, 1), (1, 40, 55, 2, 32, 17, 8, 21, 1, 0),
    (2, 96, 128, 6, 128, 32, 16, 16, 0, 1), (1, 160, 176, 12, 64, 16, 8, 8, 0, 1), (1, 3, 40, 1, 64, 32, 1, 7, 0, 1), (1, 33, 40, 150, 32, 32, 1, 7, 0, 1),
    # a label that changes between two tiles: windows of two parts, a tile a unit (16 slots to a row), and pairs of tiles of one part and of both (32)
    (1, 16, 64, 3, 64, 16, 8, 8, 0, 1), (2, 30, 50, 2, 128, 15, 7, 3, 0, 0), (1, 48, 50, 2, 32, 24, 12, 5, 0, 1), (1, 64, 96, 30, 64, 32, 16, 16, 0, 1), (1, 64, 96, 30, 128, 24, 4, 0, 0, 0),
]


@pytest.mark.parametrize("dtype,spread", [(torch.bfloat16, 25.0), (torch.float16, 500.0)], ids=["bf16", "fp16_wide_bias"])
@pytest.mark.parametrize("case", CASES, ids=["_".join(map(str, c)) for c in CASES])
def test_window_forward(case, dtype, spread):
    cfg = small_config("window_forward", *case)
    x = {k: v.to(dtype) if v.dtype == torch.bfloat16 else v * spread for k, v in make_inputs(cfg).items()}
    xg = {k: v.cuda() for k, v in x.items()}
    o, lse = terra.terra_swin_attn_fwd(terra.make_desc(cfg, dtype=dtype), xg["q"], xg["k"], xg["v"], xg["bias"])
    terra.terra_swin_check()
    ref_o, ref_lse = oracle.attn_fwd(cfg, x["q"], x["k"], x["v"], x["bias"].double().numpy())
    tok = oracle.selection_tokens(cfg, None)
    gate("o", gpu_rows(o, cfg, tok), ref_o)
    gate("lse", gpu_rows(lse, cfg, tok), ref_lse)
