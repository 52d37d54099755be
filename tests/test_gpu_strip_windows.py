"""Window sides 33 .. 128 in strips of 32 slots, forward and backward: sides around the strips' edges, windows truncated to one, two and three
strips, the seam on a strip's edge and inside one (head dim 32: at an odd token too), mask labels that change inside a tile of three strips to
a row, windows whose key tiles several CTAs share and gangs that take several windows.  Against the oracle."""
import pytest
import torch

import oracle
import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config
from tests._parity import gate, gpu_rows

pytestmark = pytest.mark.gpu

CASES = [
    # B, H, W, heads, head_dim, window, shift_h, shift_w, periodic_h, periodic_w
    (1, 33, 33, 1, 64, 33, 0, 0, 1, 1), (1, 40, 70, 2, 32, 33, 5, 16, 0, 1), (2, 64, 64, 1, 128, 64, 20, 32, 0, 0), (1, 70, 90, 1, 32, 65, 31, 25, 0, 1),
    (1, 96, 100, 1, 64, 96, 50, 33, 0, 0), (1, 45, 230, 1, 128, 100, 3, 65, 1, 1), (1, 128, 30, 1, 64, 128, 64, 7, 0, 0), (1, 3, 128, 2, 32, 128, 1, 64, 0, 1),
    (3, 35, 140, 7, 64, 40, 20, 20, 0, 1), (1, 130, 66, 3, 128, 64, 32, 16, 0, 1), (1, 34, 1, 1, 128, 128, 0, 0, 0, 1),
    # on the register tiles, forward or in both directions: windows that fill little of their strips
    (1, 68, 70, 2, 32, 34, 17, 9, 0, 1), (3, 64, 3, 2, 64, 64, 20, 1, 0, 1), (2, 8, 8, 1, 128, 40, 4, 0, 1, 0), (1, 5, 60, 2, 32, 64, 2, 7, 0, 0),
]

# gangs that take one window after another, more than their ring has slabs (tests/test_onepass_plan.py), whole ones, ones of two parts and truncated ones
GANGS = [(1, 12, 64, 200, 32, 64, 6, 32, 0, 1), (1, 12, 66, 150, 128, 64, 6, 32, 0, 1), (1, 24, 80, 100, 128, 40, 12, 20, 0, 1), (2, 20, 70, 75, 64, 64, 10, 20, 0, 0)]


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "fp16"])
@pytest.mark.parametrize("case", CASES + GANGS, ids=["_".join(map(str, c)) for c in CASES + GANGS])
def test_strip_windows(case, dtype):
    cfg = small_config("strips", *case)
    x = {k: v.to(dtype) if v.dtype == torch.bfloat16 else v * 25.0 for k, v in make_inputs(cfg).items()}
    xg = {k: v.cuda() for k, v in x.items()}
    d = terra.make_desc(cfg, dtype=dtype)
    o, lse = terra.terra_swin_attn_fwd(d, xg["q"], xg["k"], xg["v"], xg["bias"])
    got = terra.terra_swin_attn_bwd(d, xg["q"], xg["k"], xg["v"], xg["bias"], o, lse, xg["do"])
    again = terra.terra_swin_attn_bwd(d, xg["q"], xg["k"], xg["v"], xg["bias"], o, lse, xg["do"])
    terra.terra_swin_check()
    table = x["bias"].double().numpy()
    ref_o, ref_lse = oracle.attn_fwd(cfg, x["q"], x["k"], x["v"], table)
    ref = oracle.attn_bwd(cfg, x["q"], x["k"], x["v"], x["do"], table)
    tok = oracle.selection_tokens(cfg, None)
    gate("o", gpu_rows(o, cfg, tok), ref_o)
    gate("lse", gpu_rows(lse, cfg, tok), ref_lse)
    for i, name in enumerate(("dq", "dk", "dv", "dbias")):
        gate(name, gpu_rows(got[i], cfg, tok) if i < 3 else got[i].cpu().double().numpy(), ref[i])
        assert i == 3 or torch.equal(got[i], again[i])               # sums in a fixed order, whichever CTAs add


def test_strips_under_capture():
    cfg = small_config("strips", 1, 70, 130, 2, 64, 64, 32, 32, 0, 1)
    x = {k: v.cuda() for k, v in make_inputs(cfg).items()}
    d = terra.make_desc(cfg)
    o, lse = terra.terra_swin_attn_fwd(d, x["q"], x["k"], x["v"], x["bias"])
    ref = terra.terra_swin_attn_bwd(d, x["q"], x["k"], x["v"], x["bias"], o, lse, x["do"])
    grads = [torch.empty_like(t) for t in ref]
    workspace = torch.empty(terra.terra_swin_workspace_bytes(d, True), dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        terra.terra_swin_attn_bwd(d, x["q"], x["k"], x["v"], x["bias"], o, lse, x["do"], dq=grads[0], dk=grads[1], dv=grads[2], dbias=grads[3], workspace=workspace)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    for i in range(3):
        assert torch.equal(grads[i], ref[i])
    assert (grads[3] - ref[3]).norm() <= 1e-5 * ref[3].norm()        # float atomics: 32-bit sums in another order


# windows of one key tile, which no gang shares, and of two (head dim 32: with a slab, unlike below side 33), with fewer and more windows than gangs
TIGHT = [(1, 4, 32, 8, 64, 64, 2, 7, 0, 1), (1, 1, 100, 3, 128, 64, 0, 32, 0, 1), (1, 4, 32, 2, 32, 33, 0, 0, 0, 1),
         (1, 4, 64, 2, 32, 64, 2, 32, 0, 1), (1, 8, 30, 3, 32, 48, 4, 0, 0, 1), (1, 4, 5000, 12, 32, 64, 2, 32, 0, 1)]


@pytest.mark.parametrize("case", TIGHT, ids=["_".join(map(str, c)) for c in TIGHT])
def test_nothing_is_written_behind_the_workspace(case):
    """Both calls with exactly the workspace they ask for, inside a larger buffer."""
    cfg = small_config("strips", *case)
    x = make_inputs(cfg)
    xg = {k: v.cuda() for k, v in x.items()}
    d = terra.make_desc(cfg)
    need = [terra.terra_swin_workspace_bytes(d, backward) for backward in (False, True)]
    guard = 1 << 20
    buf = torch.full((2 * guard + max(need),), 0xA5, dtype=torch.uint8, device="cuda")

    def workspace(n):
        buf.fill_(0xA5)
        return buf[guard:guard + n]

    def untouched(n):
        return bool((buf[:guard] == 0xA5).all()) and bool((buf[guard + n:] == 0xA5).all())

    o, lse = terra.terra_swin_attn_fwd(d, xg["q"], xg["k"], xg["v"], xg["bias"], workspace=workspace(need[0]))
    assert untouched(need[0])
    got = terra.terra_swin_attn_bwd(d, xg["q"], xg["k"], xg["v"], xg["bias"], o, lse, xg["do"], workspace=workspace(need[1]))
    assert untouched(need[1])
    terra.terra_swin_check()
    table = x["bias"].double().numpy()
    ref_o, ref_lse = oracle.attn_fwd(cfg, x["q"], x["k"], x["v"], table)
    ref = oracle.attn_bwd(cfg, x["q"], x["k"], x["v"], x["do"], table)
    tok = oracle.selection_tokens(cfg, None)
    gate("o", gpu_rows(o, cfg, tok), ref_o)
    gate("lse", gpu_rows(lse, cfg, tok), ref_lse)
    for i, name in enumerate(("dq", "dk", "dv", "dbias")):
        gate(name, gpu_rows(got[i], cfg, tok) if i < 3 else got[i].cpu().double().numpy(), ref[i])
