"""The forward on complete windows of side 64 and 128 without mask labels, which have a kernel of their own where every SM gets more than a pair
of query tiles: on both sides of that line, seams inside windows, whole-window shifts, packed tensors and a bias table too wide for the bound on a row's
maximum.  A selection of windows against the oracle."""
import pytest
import torch

import oracle
import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config
from tests._parity import gate, gpu_rows

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, W, heads, head_dim, window, shift_h, shift_w, periodic_h, periodic_w; own kernel
    ((1, 64, 448, 2, 128, 64, 0, 40, 0, 1), True), ((1, 64, 448, 2, 128, 64, 0, 36, 0, 1), False), ((1, 64, 128, 2, 128, 64, 64, 64, 0, 0), False),
    ((2, 128, 192, 1, 128, 64, 64, 128, 0, 0), True), ((2, 128, 256, 1, 128, 64, 32, 0, 0, 1), False), ((1, 128, 384, 1, 128, 128, 0, 64, 0, 1), True),
    ((1, 64, 640, 1, 64, 64, 24, 24, 1, 1), True),
]


def _own(desc, cfg):
    per_head = 4 * ((2 * cfg.window - 1) * 2 * cfg.window + 4)
    return terra.terra_swin_workspace_bytes(desc, False) == -(-cfg.heads * per_head // 256) * 256


@pytest.mark.parametrize("dtype,spread", [(torch.bfloat16, 25.0), (torch.float16, 500.0)], ids=["bf16", "fp16_wide_bias"])
@pytest.mark.parametrize("case,own", CASES, ids=["_".join(map(str, c[0])) for c in CASES])
def test_complete_windows(case, own, dtype, spread):
    cfg = small_config("complete", *case)
    x = {k: v.to(dtype) if v.dtype == torch.bfloat16 else v * spread for k, v in make_inputs(cfg).items()}
    xg = {k: v.cuda() for k, v in x.items()}
    d = terra.make_desc(cfg, dtype=dtype)
    assert _own(d, cfg) == own
    o, lse = terra.terra_swin_attn_fwd(d, xg["q"], xg["k"], xg["v"], xg["bias"])
    op, lsep = terra.terra_swin_attn_fwd_packed(d, torch.stack((xg["q"], xg["k"], xg["v"]), dim=3).contiguous(), xg["bias"])
    terra.terra_swin_check()
    assert torch.equal(o, op) and torch.equal(lse, lsep)
    windows = cfg.B * (cfg.H // cfg.window) * (cfg.W // cfg.window)
    sel = [0, windows - 1][cfg.window // 128:]
    ref_o, ref_lse = oracle.attn_fwd(cfg, x["q"], x["k"], x["v"], x["bias"].double().numpy(), sel=sel)
    tok = oracle.selection_tokens(cfg, sel)
    gate("o", gpu_rows(o, cfg, tok), ref_o)
    gate("lse", gpu_rows(lse, cfg, tok), ref_lse)
