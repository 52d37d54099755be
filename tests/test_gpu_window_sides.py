"""Window sides on both sides of the lines that the forward's dispatch draws between the dense register tiles and the slots of 16 or 32 to
a window row, on a ragged grid with a seam and a mask.  Against the oracle."""
import pytest
import torch

import oracle
import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config
from tests._parity import gate, gpu_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "fp16"])
@pytest.mark.parametrize("head_dim,side", [(32, s) for s in (22, 23, 24, 25, 26, 27)] + [(64, s) for s in (11, 12, 16, 17, 18)] + [(128, 9), (128, 17)])
def test_window_side(head_dim, side, dtype):
    cfg = small_config("window_side", 1, 2 * side + 5, 2 * side + 3, 2, head_dim, side, side // 2, side // 2, 0, 1)
    x = {k: v.to(dtype) if v.dtype == torch.bfloat16 else v * 25.0 for k, v in make_inputs(cfg).items()}
    xg = {k: v.cuda() for k, v in x.items()}
    o, lse = terra.terra_swin_attn_fwd(terra.make_desc(cfg, dtype=dtype), xg["q"], xg["k"], xg["v"], xg["bias"])
    terra.terra_swin_check()
    ref_o, ref_lse = oracle.attn_fwd(cfg, x["q"], x["k"], x["v"], x["bias"].double().numpy())
    tok = oracle.selection_tokens(cfg, None)
    gate("o", gpu_rows(o, cfg, tok), ref_o)
    gate("lse", gpu_rows(lse, cfg, tok), ref_lse)


@pytest.mark.parametrize("side,windows", [(22, False), (23, True), (24, True), (25, False), (26, False), (27, True)])
def test_which_kernel_takes_head_dim_32(side, windows):
    cfg = small_config("window_side", 1, 2 * side, 2 * side, 2, 32, side, side // 2, side // 2, 0, 1)
    x = {k: v.cuda() for k, v in make_inputs(cfg).items()}
    terra.profile_enable(True)
    terra.terra_swin_attn_fwd(terra.make_desc(cfg), x["q"], x["k"], x["v"], x["bias"])
    torch.cuda.synchronize()
    names = [name for name, _ in terra.profile_read()]
    terra.profile_enable(False)
    assert ("swin_fwd_win_kernel" in names) == windows, names
