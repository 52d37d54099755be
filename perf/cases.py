"""Performance cases of the shifted-window attention block: what a user's program calls, over the sizes it calls it with.

A case is one forward, one backward or one training step (forward, then backward) of the block on a token grid, through
the package's binding.  The listed sizes are the repository's own configurations (`workloads.CONFIGS`), the ragged and
unpadded grids of the same field, and a regional grid of a few windows; `draw` gives more of the same ranges.

Fields: `call` ("forward", "backward", "step"), the descriptor's geometry, `dtype` ("bf16", "fp16"), `packed` (q, k, v as one
[B, H, W, 3, heads, head_dim] tensor of a fused projection) and `keep` (the program hands in its output buffers and
workspace, as a serving loop does; otherwise each call allocates its outputs, as an autograd function does).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.accounting import work as _accounting
from paper_2608_15211_b200.workloads import CONFIGS

_DTYPES = {"bf16": torch.bfloat16, "fp16": torch.float16}


def _case(name, call, B, H, W, heads, head_dim, window, shift_h, shift_w, *, periodic_h=0, periodic_w=1, dtype="bf16",
          packed=False, keep=False):
    out = {} if name is None else {"name": name}
    out.update(call=call, B=B, H=H, W=W, heads=heads, head_dim=head_dim, window=window, shift_h=shift_h, shift_w=shift_w,
               periodic_h=periodic_h, periodic_w=periodic_w, dtype=dtype, packed=packed, keep=keep)
    return out


def _config(name, config, call, **options):
    c = CONFIGS[config]
    return _case(name, call, c.B, c.H, c.W, c.heads, c.head_dim, c.window, c.shift_h, c.shift_w,
                 periodic_h=c.periodic_h, periodic_w=c.periodic_w, **options)


def listed():
    return [
        # one block of a small forecaster answering a request: 32 windows, all latency and launch
        _config("cfg1_forward", "cfg1", "forward", keep=True),
        # a training step on a regional grid that fits no window: 2 samples, 6 ragged windows each
        _case("regional_step", "step", 2, 30, 40, 3, 32, 16, 8, 8),
        # a training step of a shallow stage with the classic 8 x 8 windows
        _config("cfg2_step", "cfg2", "step"),
        # inference and the backward pass of the global quarter-million-window grid at patch 4
        _config("cfg3_forward", "cfg3", "forward", keep=True),
        _config("cfg3_backward", "cfg3", "backward"),
        # training with 32 x 32 windows at head dim 64
        _config("cfg4_step", "cfg4", "step"),
        # the fine patch (2 rollout samples, 14 x 14 windows): the largest tensors
        _config("cfg5_step", "cfg5", "step"),
        # the paper's small model in its own precision, from a fused QKV projection
        _config("tv_small_step", "tv_small", "step", dtype="fp16", packed=True),
        # the unshifted sibling block of the same grid with 16 x 16 windows
        _case("w16_d128_step", "step", 1, 288, 544, 8, 128, 16, 0, 0, packed=True),
        # 32 x 32 windows on the grid as it is (510 x 1080 tokens sampled by 2), not padded to complete windows
        _case("ragged_w32_step", "step", 1, 255, 540, 12, 64, 32, 16, 16),
        # the paper's large model: 64 heads of 128 channels
        _config("tv_large_step", "tv_large", "step"),
        # the window-assignment study's largest window, in the paper's precision: 16384 tokens attend to each other
        _config("tv_small_w128_step", "tv_small_w128", "step", dtype="fp16"),
    ]


def draw(rng):
    """Another block of these ranges: grids of 10^3 to 10^6 tokens about twice as wide as high, half of them complete windows."""
    while True:
        head_dim = rng.choice([32, 32, 64, 128])
        window = rng.choice([8, 8, 16, 16, 32, 32, rng.randint(4, 15), rng.randint(9, 31), rng.choice([64, 128])])
        tokens = math.exp(rng.uniform(math.log(1e3), math.log(1e6)))
        H = max(3, round(math.sqrt(tokens / 2) * math.exp(rng.uniform(-0.3, 0.3))))
        W = max(3, round(tokens / H))
        if rng.random() < 0.5:
            H, W = max(1, round(H / window)) * window, max(1, round(W / window)) * window
        heads = round(math.exp(rng.uniform(0.0, math.log(min(64, 4096 // head_dim)))))
        shift = rng.choice([0, window // 2, window // 2])
        case = _case(None, rng.choice(["forward", "backward", "step", "step"]), rng.choice([1, 1, 2]), H, W, heads, head_dim, window,
                     shift % H, shift % W, periodic_w=rng.choice([0, 1, 1, 1]), dtype=rng.choice(["bf16", "bf16", "fp16"]),
                     packed=rng.random() < 0.3, keep=rng.random() < 0.3)
        cost = work(case)
        if cost["flops"] <= 2.5e12 and cost["bytes"] <= 6e9:      # a fraction of the largest listed ones
            return case


def prepare(case, seed):
    """Activations and upstream gradient N(0, 1), bias table N(0, 0.02^2): projected, normalised Swin activations."""
    c = SimpleNamespace(**case)
    dtype = _DTYPES[c.dtype]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    grid = (c.B, c.H, c.W)
    row = (c.heads, c.head_dim)

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=dtype)

    desc = terra.make_desc(c, dtype=dtype)
    qkv = (normal(*grid, 3, *row),) if c.packed else tuple(normal(*grid, *row) for _ in range(3))
    s = SimpleNamespace(call=c.call, packed=c.packed, desc=desc, qkv=qkv)
    s.bias = 0.02 * torch.randn(((2 * c.window - 1) ** 2, c.heads), generator=gen, device="cuda", dtype=torch.float32)
    s.d_o = None if c.call == "forward" else normal(*grid, *row)
    s.fwd, s.bwd = {}, {}
    if c.keep:
        both = max(terra.terra_swin_workspace_bytes(desc, False), terra.terra_swin_workspace_bytes(desc, True), 16)
        workspace = torch.empty(both, dtype=torch.uint8, device="cuda")
        s.fwd = {"o": torch.empty((*grid, *row), dtype=dtype, device="cuda"), "workspace": workspace,
                 "lse": torch.empty((*grid, c.heads), dtype=torch.float32, device="cuda")}
        s.bwd = {n: torch.empty_like(s.qkv[0]) for n in (("dqkv",) if c.packed else ("dq", "dk", "dv"))}
        s.bwd.update(dbias=torch.empty_like(s.bias), workspace=workspace)
    s.saved = _forward(s) if c.call == "backward" else None
    return s


def _forward(s):
    forward = terra.terra_swin_attn_fwd_packed if s.packed else terra.terra_swin_attn_fwd
    return forward(s.desc, *s.qkv, s.bias, **s.fwd)


def _backward(s, o, lse):
    backward = terra.terra_swin_attn_bwd_packed if s.packed else terra.terra_swin_attn_bwd
    return backward(s.desc, *s.qkv, s.bias, o, lse, s.d_o, **s.bwd)


def run(s):
    if s.call == "forward":
        return _forward(s)
    if s.call == "backward":
        return _backward(s, *s.saved)
    o, lse = _forward(s)
    return (o, lse, *_backward(s, o, lse))


def work(case):
    """Each call's inputs once and outputs once; 4 d operations per allowed pair forward, 10 d backward (S anew from q and k)."""
    c = SimpleNamespace(**case)
    c.tokens = c.B * c.H * c.W
    a = _accounting(c)
    table = 4 * (2 * c.window - 1) ** 2 * c.heads
    out = {"bytes": 0, "flops": 0}
    if c.call != "backward":
        out["bytes"] += a["bytes_fwd"] + table
        out["flops"] += a["flop_fwd"]
    if c.call != "forward":
        out["bytes"] += a["bytes_bwd"] + a["tensor_bytes"] + 2 * table       # o is read as well
        out["flops"] += a["flop_bwd_fa"]
    return out


def tolerance(case):
    """Probabilities and their gradients are rounded to the activations' type before they are multiplied: 8 bits of bf16, 11 of fp16."""
    return {"rel": 1e-2, "max": 0.3} if case["dtype"] == "bf16" else {"rel": 2e-3, "max": 0.1}
