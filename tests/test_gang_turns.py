"""The turns of the CTAs that share a window's key tiles in the one-pass backward, on the CPU: for every chunk of queries the tiles' places in
the order of the adds are 0 .. tiles - 1, and CTAs that go through their tiles and chunks as the kernel does never wait for one another in a
circle.  And where a window is taken as two parts, no tile holds rows of both."""
import pytest


def _place(kt, chunk, tiles, gang, rotate):
    """attn_bwd_onepass.cu, `place`."""
    if not rotate:
        return kt
    n = min(gang, tiles)
    j = kt % n
    start = kt - j
    in_round = min(n, tiles - start)
    r = min(in_round - 1, ((chunk + 1) * n - 1) // tiles) - j
    return start + (r + in_round if r < 0 else r)


def _first_chunk(kt, tiles, gang, rotate):
    ranks = min(gang, tiles)
    return kt % ranks * tiles // ranks if rotate else 0


@pytest.mark.parametrize("rotate", [False, True])
@pytest.mark.parametrize("gang", [2, 3, 4, 7, 9, 16, 37, 64, 74, 148])
def test_turns(gang, rotate):
    for tiles in (2, 3, 4, 5, 8, 13, 16, 31, 32, 64, 97, 128):
        for chunk in range(tiles):
            assert sorted(_place(kt, chunk, tiles, gang, rotate) for kt in range(tiles)) == list(range(tiles))
        # every CTA's events in its order; an event waits for the one a place before it
        left = [[(kt, (i + _first_chunk(kt, tiles, gang, rotate)) % tiles) for kt in range(cta, tiles, gang) for i in range(tiles)] for cta in range(gang)]
        done, at = [0] * tiles, [0] * gang
        moved = True
        while moved:
            moved = False
            for cta in range(gang):
                while at[cta] < len(left[cta]) and _place(*left[cta][at[cta]], tiles, gang, rotate) == done[left[cta][at[cta]][1]]:
                    done[left[cta][at[cta]][1]] += 1
                    at[cta] += 1
                    moved = True
        assert done == [tiles] * tiles


def _part_tiles(ha, eh, row_slots):
    """win_tiles.cuh, `part_tiles`."""
    return ha * row_slots // 128 if 0 < ha < eh and ha * row_slots % 128 == 0 else 0


@pytest.mark.parametrize("row_slots", [16, 32, 64, 96, 128])
def test_parts_end_on_a_tile(row_slots):
    for eh in range(1, 129):
        for ha in range(-3, 132):
            first = _part_tiles(ha, eh, row_slots)
            if first:
                rows = [[slot // row_slots for slot in range(128 * t, min(128 * (t + 1), eh * row_slots))] for t in range(-(-eh * row_slots // 128))]
                assert all(r < ha for tile in rows[:first] for r in tile) and all(r >= ha for tile in rows[first:] for r in tile)
