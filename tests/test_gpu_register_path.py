"""The register-tile kernels where the dispatch prefers others (TERRA_REGISTER_PATH=1, read once, hence a process of its own), against the
oracle: sides above 32 on grids so low or narrow that a window holds no more than 256 tokens, complete along its width and not."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import oracle
import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import make_inputs, small_config
from tests._parity import gate, gpu_rows
for case in ((2, 1, 200, 3, 32, 100, 0, 50, 0, 1), (2, 4, 128, 2, 64, 64, 2, 32, 0, 1), (1, 7, 66, 2, 128, 33, 3, 5, 0, 0), (1, 70, 2, 1, 64, 40, 20, 1, 0, 1)):
    cfg = small_config("register", *case)
    x = make_inputs(cfg)
    xg = {k: v.cuda() for k, v in x.items()}
    d = terra.make_desc(cfg)
    assert terra.terra_swin_workspace_bytes(d, False) == 0
    o, lse = terra.terra_swin_attn_fwd(d, xg["q"], xg["k"], xg["v"], xg["bias"])
    got = terra.terra_swin_attn_bwd(d, xg["q"], xg["k"], xg["v"], xg["bias"], o, lse, xg["do"])
    table = x["bias"].double().numpy()
    ref_o, ref_lse = oracle.attn_fwd(cfg, x["q"], x["k"], x["v"], table)
    ref = oracle.attn_bwd(cfg, x["q"], x["k"], x["v"], x["do"], table)
    tok = oracle.selection_tokens(cfg, None)
    gate("o", gpu_rows(o, cfg, tok), ref_o)
    gate("lse", gpu_rows(lse, cfg, tok), ref_lse)
    for i, name in enumerate(("dq", "dk", "dv", "dbias")):
        gate(name, gpu_rows(got[i], cfg, tok) if i < 3 else got[i].cpu().double().numpy(), ref[i])
print("parity")
"""


def test_register_tiles_above_side_32():
    proc = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, env={**os.environ, "TERRA_REGISTER_PATH": "1", "PYTHONPATH": ROOT},
                          capture_output=True, text=True, timeout=300)
    assert proc.returncode == 0 and "parity" in proc.stdout, proc.stdout[-2000:] + proc.stderr[-4000:]
