"""The window forward's pool of shared-memory slots, on the CPU: a wait names an mbarrier phase by parity, so a role may wait for a slot's
fill only when it knows that the slot's fill before has landed; otherwise the wait is over at once and the role works on whatever
the slot holds.  The slots' order is stepped through as the kernel's roles do it, with the waits that the source has."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15211_b200", "csrc", "attn_fwd_win.cu")


def _section(begin, end):
    text = open(SOURCE).read()
    return text[text.index(begin):text.index(end)]


def _score_waits():
    """Which fills the score warp waits for."""
    text = _section("- S = Q K^T", "- O += P V")
    return {"Q0": "wait_full(s_q[0])" in text, "Q1": "wait_full(s_q[1])" in text, "K": "wait_full(sk)" in text, "V": "wait_full(sv)" in text}


def _slots(head_dim, row_slots):
    m = re.search(r"kSlots = D == 128 \? \(RW == 16 \? (\d+) : (\d+)\) : D == 64 \? (\d+) : (\d+);", open(SOURCE).read())
    return int(m[1 if row_slots == 16 else 2]) if head_dim == 128 else int(m[3 if head_dim == 64 else 4])


def _fills(slots, units):
    """(slot, fill, unit, chunk) in the order of the loads; `units`: (chunks, query tiles) each."""
    queue, out = list(range(slots)), []

    def take():
        s = queue.pop(0)
        queue.insert(slots - 3, s)
        return s

    for u, (chunks, tiles) in enumerate(units):
        q0, q1 = queue.pop(0), queue.pop(0)
        out.append((q0, "Q0", u, 0))
        for c in range(chunks):
            out.append((take(), "K", u, c))
            if c == 0 and tiles == 2:
                out.append((q1, "Q1", u, 0))
            out.append((take(), "V", u, c))
        queue += [q0, q1]
    return out


RUNS = [[(8, 2)] * 20, [(2, 2)] * 20, [(1, 1)] * 9, [(5, 2), (5, 2), (5, 1)] * 6, [(1, 2), (2, 2), (1, 1), (8, 2), (3, 1)] * 5, [(6, 2), (1, 1), (7, 2)] * 6]


@pytest.mark.parametrize("units", RUNS, ids=range(len(RUNS)))
@pytest.mark.parametrize("head_dim,row_slots", [(32, 32), (64, 16), (64, 32), (128, 16), (128, 32)])
def test_a_fill_is_waited_for_behind_the_one_before(head_dim, row_slots, units):
    fills, waits = _fills(_slots(head_dim, row_slots), units), _score_waits()
    last = {}
    for slot, fill, unit, chunk in fills:
        before = last.get(slot)
        if before is not None:
            # the score warp: a fill before is known to have landed if it has waited for it
            if waits[fill]:
                assert waits[before[0]], f"scores wait for {fill} of unit {unit}, chunk {chunk}, behind {before}, which nothing has waited for"
            # the product warp waits for V alone: Q and K have landed where it has issued a product of their scores
            if fill == "V" and before[0] != "V":
                assert before[1] < unit or (before[0] == "K" and before[2] < chunk), (fill, unit, chunk, before)
        last[slot] = (fill, unit, chunk)
