"""The shift mask and the slots without a token exclude a key whatever the scores are: forbidden keys that outscore the allowed ones
by more than any finite penalty, empty slots against scores far below zero, a score scale that shrinks every score to nothing,
and keys that are not a number.  Every forward kernel family, both element types, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config
from tests._parity import gate, gpu_rows

pytestmark = pytest.mark.gpu

SHAPES = [
    # B, H, W, heads, head_dim, window, shift_h, shift_w, periodic_h, periodic_w
    (1, 45, 50, 2, 64, 20, 10, 10, 0, 0), (1, 96, 64, 1, 128, 32, 16, 16, 0, 1), (1, 40, 55, 2, 128, 13, 6, 5, 0, 0), (1, 48, 80, 2, 64, 16, 8, 8, 0, 0),
    (1, 60, 73, 1, 32, 24, 12, 12, 0, 0), (1, 40, 46, 2, 32, 14, 7, 7, 0, 0), (1, 24, 20, 2, 64, 8, 4, 4, 0, 0), (1, 30, 32, 2, 64, 10, 5, 5, 0, 0),
    (1, 128, 64, 1, 64, 64, 32, 8, 0, 1), (1, 50, 44, 1, 64, 40, 20, 11, 0, 0),
]
HUGE = {torch.float16: 60000.0, torch.bfloat16: 2.0 ** 60}
TINY = {torch.float16: 1e-12, torch.bfloat16: 2e-38}


def _inputs(cfg, dtype):
    x = {k: v.to(dtype) if v.dtype == torch.bfloat16 else v for k, v in make_inputs(cfg).items()}
    u, v = torch.arange(cfg.H).view(1, -1, 1, 1), torch.arange(cfg.W).view(1, 1, -1, 1)
    label = 2 * ((u < cfg.shift_h) & (cfg.periodic_h == 0)) + 1 * ((v < cfg.shift_w) & (cfg.periodic_w == 0))
    return x, label.expand(cfg.B, cfg.H, cfg.W, cfg.heads)


def _forward(cfg, dtype, x, scale=0.0):
    xg = {k: v.cuda() for k, v in x.items()}
    o, lse = terra.terra_swin_attn_fwd(terra.make_desc(cfg, scale=scale, dtype=dtype), xg["q"], xg["k"], xg["v"], xg["bias"])
    terra.terra_swin_check()
    tok = oracle.selection_tokens(cfg, None)
    return gpu_rows(o, cfg, tok), gpu_rows(lse, cfg, tok), tok


def _compare(cfg, dtype, x, scale=0.0):
    o, lse, _ = _forward(cfg, dtype, x, scale)
    ref_o, ref_lse = oracle.attn_fwd(cfg, x["q"], x["k"], x["v"], x["bias"].double().numpy(), **({"scale": scale} if scale else {}))
    gate("o", o, ref_o)
    gate("lse", lse, ref_lse)


cases = pytest.mark.parametrize("case", SHAPES, ids=["_".join(map(str, c)) for c in SHAPES])
types = pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16], ids=["bf16", "fp16"])


@types
@cases
def test_forbidden_keys_with_the_largest_scores(case, dtype):
    # channel 0: only unwrapped queries meet wrapped keys there, and the two never share a label
    cfg = small_config("forward_mask", *case)
    x, label = _inputs(cfg, dtype)
    x["q"][..., 0] = torch.where(label > 0, 0.0, HUGE[dtype]).to(dtype)
    x["k"][..., 0] = torch.where(label > 0, HUGE[dtype], 0.0).to(dtype)
    _compare(cfg, dtype, x)


@types
@cases
def test_empty_slots_against_scores_far_below_zero(case, dtype):
    # all scores of a row are equal, far below that of a slot of zeros; a power of two, so that they are exact
    cfg = small_config("forward_mask", *case)
    x, _ = _inputs(cfg, dtype)
    c = 2.0 ** 15 if dtype == torch.float16 else 2.0 ** 52
    x["q"] = torch.zeros_like(x["q"])
    x["q"][..., :8] = c
    x["k"] = -x["q"]
    x["bias"] = torch.zeros_like(x["bias"])
    _compare(cfg, dtype, x)


@types
@cases
def test_scale_that_shrinks_every_score(case, dtype):
    cfg = small_config("forward_mask", *case)
    x, _ = _inputs(cfg, dtype)
    _compare(cfg, dtype, x, TINY[dtype])


@cases
def test_a_key_that_is_not_a_number_stays_in_its_region(case):
    cfg = small_config("forward_mask", *case)
    x, label = _inputs(cfg, torch.bfloat16)
    clean, clean_lse, tok = _forward(cfg, torch.bfloat16, x)
    x["k"][0, 0, 0] = float("nan")                  # tokens of another label than this one's may not see it
    o, lse, _ = _forward(cfg, torch.bfloat16, x)
    free = (label != label[0, 0, 0, 0]).reshape(-1, cfg.heads)[torch.from_numpy(np.asarray(tok))].numpy()
    assert free.any() and np.array_equal(o[free], clean[free]) and np.array_equal(lse[free], clean_lse[free])
