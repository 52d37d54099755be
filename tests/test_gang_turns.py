"""The turns of the CTAs that share a window's key tiles in the one-pass backward, on the CPU, with the kernel's own functions (csrc/win_tiles.cuh) in
a host program: for every chunk of queries the tiles' places in the order of the adds are 0 .. tiles - 1; and gangs that go through their
windows as the kernel does (windows of two parts, a ring of slabs, turns of several dQ events, flags raised an event late) never wait in a
circle, add in the order of the places and start on a slab only when its last window has left it.  And where a window is taken as two parts,
no tile holds rows of both."""
from tests._host_program import run_host_program

PLACES = """
int main() {
    for (int gang : {2, 3, 4, 7, 9, 16, 37, 64, 74, 148})
        for (int tiles : {1, 2, 3, 4, 5, 8, 13, 16, 31, 32, 64, 97, 128})
            for (bool rotate : {false, true}) {
                for (int c = 0; c < tiles; ++c) {
                    bool seen[128] = {};
                    for (int kt = 0; kt < tiles; ++kt) {
                        const int at = gang_place(kt, c, tiles, gang, rotate);
                        if (at < 0 || at >= tiles || seen[at]) return std::printf("place of %d at %d, %d tiles, gang %d\\n", kt, c, tiles, gang), 1;
                        seen[at] = true;
                    }
                }
                for (int seq : {0, 1, 5, 100}) {
                    int taken = 0;
                    for (int member = 0; member < gang; ++member)
                        for (int kt = gang_first_tile(member, seq, gang); kt < tiles; kt += gang) {
                            const int first = gang_first_chunk(kt, tiles, gang, rotate);
                            if (kt < 0 || (seq + kt) % gang != member || first < 0 || first >= tiles) return std::printf("tile %d of member %d\\n", kt, member), 1;
                            ++taken;
                        }
                    if (taken != tiles) return std::printf("%d of %d tiles taken\\n", taken, tiles), 1;
                }
            }
    return 0;
}
"""

RUNS = """
#include <vector>
// One gang's windows, given by their parts' tiles; `per_chunk` dQ events a chunk, turns of 1 << turn_log2 events.  What attn_bwd_onepass.cu's planning
// warp deals and its read-out warps do (`turn`, `turn_done`, `signal`).
struct Tile { int part, kt, tn, q0, slab, seq, use, c0; };
static int run(const std::vector<std::vector<int>>& windows, int gang, int ring, bool rotate, int per_chunk, int turn_log2) {
    std::vector<std::vector<Tile>> todo(gang);
    std::vector<int> tiles_of;
    int seq = 0, used = 0, most = 0;
    for (const auto& window : windows) {
        int q0 = 0;
        for (int tn : window) {
            for (int m = 0; m < gang; ++m)
                for (int kt = gang_first_tile(m, seq, gang); kt < tn; kt += gang)
                    todo[m].push_back({(int)tiles_of.size(), kt, tn, q0, used % ring, seq, used / ring, gang_first_chunk(kt, tn, gang, rotate)});
            tiles_of.push_back(tn);
            seq += tn;
            used += tn > 1;
            q0 += tn;
        }
        most = std::max(most, q0);
    }
    const int events = most * per_chunk, turn = 1 << turn_log2;
    std::vector<int> flags(ring * (events + 1), 0), owner(ring * events, -1), adds(ring * events, 0);
    struct Cta { size_t tile = 0; int i = 0, pending = -1, value = 0; };
    std::vector<Cta> ctas(gang);
    bool moved = true;
    while (moved) {
        moved = false;
        for (int m = 0; m < gang; ++m) {
            Cta& c = ctas[m];
            while (c.tile < todo[m].size()) {
                const Tile& t = todo[m][c.tile];
                int* f = &flags[t.slab * (events + 1)];
                const int n = t.tn * per_chunk;
                if (t.tn > 1) {
                    if (c.i < n) {
                        const int rel = (c.i + t.c0 * per_chunk) % n, ev = rotate ? t.q0 * per_chunk + rel : rel;
                        const int at = gang_place(t.kt, rel / per_chunk, t.tn, gang, rotate);
                        if (c.pending >= 0) { flags[c.pending] = c.value; c.pending = -1; }
                        const bool starts = ev % turn == 0;
                        if (starts && at > 0 && f[ev >> turn_log2] < t.seq + at) break;
                        if (starts && at == 0 && !rotate && ev == 0 && f[events] < t.use) break;
                        // the add itself: in order, to the slab's part that this window has
                        const int cell = t.slab * events + (rotate ? t.q0 * per_chunk + rel : rel);
                        if (at == 0) { owner[cell] = t.part; adds[cell] = 0; }
                        if (owner[cell] != t.part || adds[cell] != at) return std::printf("tile %d of part %d adds out of turn\\n", t.kt, t.part), 1;
                        ++adds[cell];
                        if (at != t.tn - 1 && (rel == n - 1 || (ev + 1) % turn == 0)) {
                            c.pending = t.slab * (events + 1) + (ev >> turn_log2);
                            c.value = t.seq + at + 1;
                        }
                        ++c.i;
                        moved = true;
                        continue;
                    }
                    if (c.pending >= 0) { flags[c.pending] = c.value; c.pending = -1; }
                    if (!rotate && t.kt == t.tn - 1) f[events] = t.use + 1;
                }
                ++c.tile;
                c.i = 0;
                moved = true;
            }
        }
    }
    for (int m = 0; m < gang; ++m)
        if (ctas[m].tile < todo[m].size()) return std::printf("CTA %d of %d waits for good (ring %d, rotate %d)\\n", m, gang, ring, rotate), 1;
    return 0;
}
int main() {
    for (int gang : {2, 3, 4, 5, 7, 9, 16, 37, 74}) {
        for (int tiles : {2, 3, 5, 8, 13, 17, 32, 64})
            for (int t0 : {0, 1, tiles / 2}) {
                const std::vector<int> whole = {tiles}, two = {t0, tiles - t0}, low = {1}, odd = {std::max(1, tiles / 3)};
                const auto& x = t0 > 0 && t0 < tiles ? two : whole;
                // head dim 128: two events a chunk, turns of 256 queries (rotate: 128); else one and turns of 256 (128)
                for (int per_chunk : {1, 2}) {
                    if (run({x}, gang, 1, true, per_chunk, per_chunk - 1)) return 1;
                    for (int ring : {1, 2, 3, 6}) {
                        std::vector<std::vector<int>> many;
                        for (int i = 0; i < 3 * ring + 2; ++i) many.push_back(i % 5 == 3 ? low : i % 3 == 1 ? odd : i % 2 ? whole : x);
                        if (run(many, gang, ring, false, per_chunk, per_chunk)) return 1;
                    }
                }
            }
    }
    return 0;
}
"""

PARTS = """
int main() {
    for (int row_slots : {16, 32, 64, 96, 128})
        for (int eh = 1; eh <= 128; ++eh)
            for (int ha = -3; ha < 132; ++ha) {
                const int first = part_tiles(ha, eh, row_slots);
                for (int slot = 0; first > 0 && slot < eh * row_slots; ++slot)
                    if ((slot / 128 < first) != (slot / row_slots < ha)) return std::printf("%d slots a row, %d rows, label from %d\\n", row_slots, eh, ha), 1;
            }
    return 0;
}
"""


def test_every_tile_has_a_place_and_a_cta(tmp_path):
    run_host_program(tmp_path, PLACES)


def test_gangs_get_through_their_windows(tmp_path):
    run_host_program(tmp_path, RUNS)


def test_parts_end_on_a_tile(tmp_path):
    run_host_program(tmp_path, PARTS)
