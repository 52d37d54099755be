"""The one-pass backward kernel at the edges of its range: sides 9, 16, 17 and 32 of the two slot layouts, one and several key
tiles, truncated windows, seams that cut a window column at an odd token, columns behind the seam, windows whose key tiles are
shared by several CTAs and CTAs that take several windows.  Against the oracle."""
import pytest
import torch

import oracle
import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config
from tests._parity import gate, gpu_rows

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, W, heads, head_dim, window, shift_h, shift_w, periodic_h, periodic_w
    (1, 32, 32, 1, 64, 32, 0, 0, 1, 1), (1, 41, 50, 2, 128, 13, 6, 5, 0, 0), (2, 27, 30, 2, 64, 9, 4, 3, 0, 1), (1, 48, 80, 3, 128, 16, 0, 0, 0, 1),
    (2, 45, 50, 2, 64, 20, 10, 10, 0, 1), (1, 70, 45, 2, 64, 31, 20, 30, 0, 0), (2, 80, 70, 5, 64, 17, 8, 9, 1, 0), (1, 64, 64, 2, 32, 32, 16, 16, 0, 1),
    (1, 60, 73, 3, 32, 24, 12, 12, 0, 1), (1, 40, 55, 2, 32, 17, 8, 21, 1, 0), (1, 35, 66, 2, 128, 32, 5, 40, 0, 1), (2, 96, 128, 6, 128, 32, 16, 16, 0, 1),
    (1, 160, 176, 12, 64, 16, 8, 8, 0, 1), (1, 3, 40, 1, 64, 32, 1, 7, 0, 1),
]


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "fp16"])
@pytest.mark.parametrize("case", CASES, ids=["_".join(map(str, c)) for c in CASES])
def test_onepass_backward(case, dtype):
    cfg = small_config("onepass", *case)
    x = {k: v.to(dtype) if v.dtype == torch.bfloat16 else v * 25.0 for k, v in make_inputs(cfg).items()}
    xg = {k: v.cuda() for k, v in x.items()}
    d = terra.make_desc(cfg, dtype=dtype)
    o, lse = terra.terra_swin_attn_fwd(d, xg["q"], xg["k"], xg["v"], xg["bias"])
    got = terra.terra_swin_attn_bwd(d, xg["q"], xg["k"], xg["v"], xg["bias"], o, lse, xg["do"])
    again = terra.terra_swin_attn_bwd(d, xg["q"], xg["k"], xg["v"], xg["bias"], o, lse, xg["do"])
    terra.terra_swin_check()
    ref = oracle.attn_bwd(cfg, x["q"], x["k"], x["v"], x["do"], x["bias"].double().numpy())
    tok = oracle.selection_tokens(cfg, None)
    for i, name in enumerate(("dq", "dk", "dv", "dbias")):
        gate(name, gpu_rows(got[i], cfg, tok) if i < 3 else got[i].cpu().double().numpy(), ref[i])
        assert i == 3 or torch.equal(got[i], again[i])               # sums in a fixed order
