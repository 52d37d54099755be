"""The one-pass backward's plan over the sides and grids that it takes, on the CPU: what the kernels write into the workspace lies in it."""
import paper_2608_15211_b200 as terra
from paper_2608_15211_b200.workloads import small_config
from tests._host_program import run_host_program
from tests.test_gpu_strip_windows import GANGS

SWEEP = """
int main() {
    const int heights[] = {1, 2, 3, 4, 5, 8, 16, 33, 64, 100, 128, 130, 260}, widths[] = {1, 20, 32, 33, 64, 96, 97, 128, 129, 700, 5000};
    const int sides[] = {11, 16, 17, 32, 33, 34, 40, 64, 65, 96, 97, 128};
    long long n = 0, bad = 0;
    for (int B : {1, 3}) for (int H : heights) for (int W : widths) for (int heads : {1, 2, 3, 8, 12, 37, 64, 148}) for (int d : {32, 64, 128}) for (int w : sides) {
        terra_swin_desc desc = {B, H, W, heads, d, w, 0, 0, 0, 1, 0.f, TERRA_DTYPE_BF16};
        Geo g;
        if (resolve_attention_geo(&desc, &g) != TERRA_OK || !bwd_onepass_supported(g)) continue;
        const OnePassPlan p = bwd_onepass_plan(g);
        ++n;
        // dQ slabs: of every unit where windows are split, of every gang's ring, else of the CTAs of the launches that may run at the same time
        const int tiles = p.npad / 128;
        const bool uses = tiles > (d == 32 && !p.strips && p.split_log2 == 0 ? 2 : 1);
        const long long ctas = std::min<long long>(p.units, (d == 128 || p.strips ? 1 : 2) * kMaxCtas);
        const size_t slabs = !uses ? 0 : p.split_log2 ? p.units : p.gang > 1 ? (long long)p.gangs * p.ring : ctas, end = p.off_slabs + 4 * slabs * p.npad * d;
        const bool flags = p.off_flags >= p.off_slabs && p.off_flags + 4 * (size_t)p.flags <= p.bytes;
        if ((!flags || end > (p.flags ? p.off_flags : p.bytes)) && bad++ < 10)
            std::printf("B %d, %d x %d, %d x %d, side %d: gangs %d of %d, slabs from %zu to %zu, flags from %zu to %zu of %zu\\n", B, H, W, heads, d, w, p.gangs, p.gang,
                        p.off_slabs, end, p.off_flags, p.off_flags + 4 * (size_t)p.flags, p.bytes);
        // on fewer SMs: CTAs that fit, slabs and flags of the plan, and CTAs that start at different chunks only where no gang has a second window
        for (int ctas : {1, 2, 3, 8, 16, 37, 72, 100, 147, 148, 160}) {
            if (p.gang < 2) break;
            const GangShape s = fit_gangs(p, p.units, ctas);
            const bool fits = s.gangs >= 1 && s.gang >= 1 && s.gangs * s.gang <= ctas && s.gangs <= p.gangs && s.gang <= p.gang && (!s.rotate || s.gangs >= p.units) &&
                              (s.gang > 1 || ctas == 1) && (ctas < p.gangs * p.gang || (s.gangs == p.gangs && s.gang == p.gang && s.rotate == p.rotate));
            if (!fits && bad++ < 10) std::printf("%d CTAs for %d gangs of %d: %d of %d\\n", ctas, p.gangs, p.gang, s.gangs, s.gang);
        }
    }
    std::printf("%lld plans, %lld bad\\n", n, bad);
    return bad != 0 || n == 0;
}
"""


def test_slabs_and_flags_lie_in_the_workspace(tmp_path):
    run_host_program(tmp_path, SWEEP)


RING = """
int main(int argc, char** argv) {
    for (int i = 1; i + 9 < argc; i += 10) {
        int x[10];
        for (int j = 0; j < 10; ++j) x[j] = std::atoi(argv[i + j]);
        terra_swin_desc desc = {x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], x[8], x[9], 0.f, TERRA_DTYPE_BF16};
        Geo g;
        if (resolve_attention_geo(&desc, &g) != TERRA_OK || !bwd_onepass_supported(g)) return 1;
        const OnePassPlan p = bwd_onepass_plan(g);
        if (p.gang < 2 || p.rotate || p.units <= (long long)p.gangs * p.ring)
            return std::printf("%lld windows, gangs %d of %d, ring %d, rotate %d\\n", p.units, p.gangs, p.gang, p.ring, p.rotate), 1;
    }
    return 0;
}
"""


def test_gang_cases_go_round_their_rings(tmp_path):
    """The GPU cases of that name have more windows for every gang than it has slabs."""
    run_host_program(tmp_path, RING, *(v for case in GANGS for v in case))


def test_more_heads_than_the_tables_entries_can_be_numbered_for():
    """Head counts behind which 32 bits do not number the entries of the one-pass backward's bias tables take the register tiles, whose workspace
    is a float per token and head."""
    for window, per_head in ((128, 2 * 132 * 256), (33, 2 * 37 * 128), (32, 2 * 32 * 64)):
        most = (2**31 - 2**20) // per_head
        for heads, tables in ((most, True), (most + 1, False), (2 * most, False)):
            desc = terra.make_desc(small_config("heads", 1, 1, 2, heads, 128, window, 0, 0))
            need, delta = terra.terra_swin_workspace_bytes(desc, True), 4 * 2 * heads
            assert need > 3 * 4 * per_head * heads if tables else delta <= need < delta + 256
