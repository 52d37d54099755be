"""Workspace of the one-pass backward, on the CPU: statistics per slot pair, three bias tables, and a dQ slab per CTA of the launches that
may run at the same time (head dim 128: one launch, otherwise the masked windows' beside the others')."""
import pytest

import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.build import build
from paper_2608_15211_b200.workloads import CONFIGS

MAX_CTAS, ROW_SLOTS, LAUNCHES = 160, 32, {64: 2, 128: 1}


@pytest.mark.parametrize("name", ["cfg4", "tv_large"])
def test_workspace_holds_a_slab_per_cta(name):
    build()
    c = CONFIGS[name]
    slots = c.window * ROW_SLOTS
    items = c.B * -(-c.H // c.window) * -(-c.W // c.window) * c.heads
    stats, tables = 16 * items * slots // 2, 3 * 4 * c.heads * 2 * c.window * 2 * ROW_SLOTS
    slabs = 4 * min(items, LAUNCHES[c.head_dim] * MAX_CTAS) * slots * c.head_dim
    got = terra.terra_swin_workspace_bytes(terra.make_desc(c), True)
    assert 0 <= got - (stats + tables + slabs) <= 5 * 256
