"""The window forward's pool of shared-memory slots, on the CPU: a wait names an mbarrier phase by parity, so a role that waits on a barrier
has to wait for each of its fills; behind one that it skips and that has not landed, the next wait is over at once and the role works
on whatever the slot holds.  The slots' order is stepped through as the kernel's roles do it, with the barriers and waits of the source."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_15211_b200", "csrc", "attn_fwd_win.cu")


def _section(begin, end):
    text = open(SOURCE).read()
    return text[text.index(begin):text.index(end)]


def _barrier(fill):
    """Which of a slot's full barriers a fill completes."""
    tensor = {"Q0": "q0, (kBFull\\w*), mq", "Q1": "q1, (kBFull\\w*), mq", "K": r"sq.take\(\), (kBFull\w*), mk", "V": r"sq.take\(\), (kBFull\w*), mv"}[fill]
    return re.search(r"fill\(" + tensor, open(SOURCE).read())[1]


def _waits(section):
    """The fills that a role waits for, with the barrier it waits on."""
    names = {"wait_full(s_q[0])": "Q0", "wait_full(s_q[1])": "Q1", "wait_full(sk)": "K", "wait_full(sv)": "V"}
    found = {fill: re.search(r"bar\((kBFull\w*) \+ s\)", section)[1] for call, fill in names.items() if call in section}
    direct = re.search(r"mbar_wait_all\(bar\((kBFull\w*) \+ sv\)", section)
    return {**found, **({"V": direct[1]} if direct else {})}


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
def test_a_role_waits_for_every_fill_of_its_barriers(head_dim, row_slots, units):
    for begin, end in (("- S = Q K^T", "- O += P V"), ("- O += P V", "// teardown")):
        waits, skipped = _waits(_section(begin, end)), {}
        assert waits
        for slot, fill, unit, chunk in _fills(_slots(head_dim, row_slots), units):
            barrier = (slot, _barrier(fill))
            if waits.get(fill) == barrier[1]:
                assert barrier not in skipped, f"{fill} of unit {unit}, chunk {chunk} is waited for behind {skipped[barrier]}, which is not"
            elif barrier[1] in waits.values():
                skipped[barrier] = (fill, unit, chunk)
