// Windows as tiles of slots, loaded by tiled bulk copies (TMA) on ANY grid: shared by the window forward, the one-pass
// backward and their host sides.
//
// A window's slots are laid out RW to a window row (RW = 16 for window sides 9 .. 16, 32 for 17 .. 32): slot = RW a + b.
// Sides 33 .. 128 (ST): a window row is `ns` strips of 32 slots (as many as the window's width needs), row after row: unit = ns a +
// (strip), slot = 32 unit + b.  A unit is then what a window row is at sides 17 .. 32, to the copies and to the elementwise warps.
// Slots with b at or beyond the window's width, or a at or beyond its height, hold no token; the copies fill them with
// zeros.  A tensor is described as [heads * d channels][w columns of a window][window columns][token rows], based at
// the first token of the shifted frame, so that a box of RW columns reads past the w columns of its window only into
// the zero fill.  64 slots (64 / RW window rows) of one channel part are one copy (4 or 8 KB) wherever the rows are
// consecutive.  What the description cannot hold gets maps of its own: window columns that lie wholly behind the
// longitude seam, the one that the seam cuts (two pieces per window row) and a truncated last column.
#pragma once
#include <cuda.h>

#include <type_traits>

#include "swin_common.cuh"
#include "tc_common.cuh"

namespace terra {

struct WinMaps {
    CUtensorMap group;       // columns in front of the seam, 64 / RW window rows per copy (ST: 64 slots of one)
    CUtensorMap row;         // the same, one window row per copy (ST: a strip of one; so below)
    CUtensorMap wrapped;     // columns behind the seam, one window row
    CUtensorMap seam_a;      // the column cut by the seam: its tokens in front of the seam ...
    CUtensorMap seam_b;      // ... and behind it, up to slot RW (ST: both of the strip that it cuts)
    CUtensorMap last;        // a truncated last column (when the seam does not cut it)
};

// (apart: with them in every kernel's arguments, four tensors' maps leave the 4 KB that a launch passes at once, and a small call took 3 us longer)
struct WinStripMaps : WinMaps {
    CUtensorMap seam_fa;     // ST: the whole strips in front of the seam ...
    CUtensorMap seam_fb;     // ... and behind it
};

struct WinCols {
    int seam;                // window column cut by the seam (-1: none), n1 of its tokens lie in front of it
    int n1;
    int first_wrapped;       // columns >= this one start behind the seam
    int last;                // truncated last column that needs the map of its own (-1: none)
    int skip;                // 64-byte rows and an odd n1: slot n1 of the seam column is copied by the loading warp itself
                             // (a bulk copy must start on a 128-byte boundary), seam_b starts one token later
};

constexpr int kMaxOnePassW = 32, kMaxWinW = 128;
inline int win_row_slots(const Geo& g) { return g.w <= 16 ? 16 : 32; }
inline bool win_strips(const Geo& g) { return g.w > 32; }

// ST: strips of a window that is `ew` wide, and the row of a unit (u / ns for u < 2^14)
__host__ __device__ __forceinline__ int strips_of(int ew) { return (ew + 31) >> 5; }
__device__ __forceinline__ int unit_row(int u, int ns) {
    const unsigned inv = ns == 1 ? 65536u : ns == 2 ? 32768u : ns == 3 ? 21846u : 16384u;
    return (int)(((unsigned)u * inv) >> 16);
}

// host: what the windows of a (sample, head) hold in blocks of 64 x 64 pairs, as register tiles count them (`dense`) and in strips (`strips`: 64
// keys x 128 queries are two, and a 128-slot tile costs four of its own)
struct StripWork { long long dense, strips; };
inline StripWork strip_work(const Geo& g) {
    StripWork x = {0, 0};
    const int rows[2] = {g.H / g.w, g.H % g.w ? 1 : 0}, cols[2] = {g.W / g.w, g.W % g.w ? 1 : 0};
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) {
            const long long eh = i ? g.H % g.w : g.w, ew = j ? g.W % g.w : g.w, n = (long long)rows[i] * cols[j];
            const long long blocks = (eh * ew + 63) / 64, units = eh * ((ew + 31) / 32), tiles = (units + 3) / 4;
            x.dense += n * blocks * blocks;
            x.strips += n * 2 * tiles * ((units + 1) / 2 + 2);
        }
    return x;
}

// host (attn_fwd_tc.cu, beside the driver's encoder)
bool encode_win_map(CUtensorMap* map, const Geo& g, const void* base, int token_stride, int nb, int ncols, int box_ch, int box_b, int box_rows);
// host (attn_bwd_onepass.cu): false if the driver's encoder is not available
bool make_win_cols(WinCols* c, const Geo& g);
bool make_win_maps(WinMaps* m, const WinCols& c, const Geo& g, const void* base, int token_stride);
bool make_win_maps(WinStripMaps* m, const WinCols& c, const Geo& g, const void* base, int token_stride);

// device: whether the `groups` 64-slot groups from window row `a0` on are one copy each (map `group`)
template <int RW>
__device__ __forceinline__ bool win_group_whole(const WinCols& c, const Geo& g, int wr, int wc, int eh, int a0, int groups) {
    int u = wr * g.w + a0 + g.sh;
    if (u >= g.H) u -= g.H;
    return wc != c.seam && wc < c.first_wrapped && wc != c.last && a0 + groups * (64 / RW) <= eh && u + groups * (64 / RW) <= g.H;
}

// device: the RW slots of window row `a`, channels [ch, ch + part) of every token, to `dst` (rows of ROWB bytes); the bytes are
// counted on `bar` (RW * ROWB, less ROWB for a seam column with c.skip).  A lane per row: a lane's copies follow one another at
// 250 cycles each, those of different lanes overlap.
template <int RW, int ROWB>
__device__ __forceinline__ void load_win_row(const WinMaps& m, const WinCols& c, uint32_t dst, const Geo& g, int b, int wr, int wc, int eh,
                                             int a, int ch, uint32_t bar) {
    int u = wr * g.w + a + g.sh;
    if (u >= g.H) u -= g.H;
    const int y = a < eh ? b * g.H + u : g.B * g.H;       // behind the last row: zeros
    if (wc == c.seam) {
        tc::tma_load_4d(dst, &m.seam_a, ch, 0, 0, y, bar);
        if (c.n1 + c.skip < RW) tc::tma_load_4d(dst + (c.n1 + c.skip) * ROWB, &m.seam_b, ch, c.skip, 0, y, bar);
    } else if (wc == c.last) {
        tc::tma_load_4d(dst, &m.last, ch, 0, 0, y, bar);
    } else if (wc >= c.first_wrapped) {
        tc::tma_load_4d(dst, &m.wrapped, ch, 0, wc - c.first_wrapped, y, bar);
    } else {
        tc::tma_load_4d(dst, &m.row, ch, 0, wc, y, bar);
    }
}

// device, ST: strip `s` of window row `a` (32 slots; see load_win_row)
template <int ROWB>
__device__ __forceinline__ void load_win_strip(const WinStripMaps& m, const WinCols& c, uint32_t dst, const Geo& g, int b, int wr, int wc, int eh,
                                               int a, int s, int ch, uint32_t bar) {
    int u = wr * g.w + a + g.sh;
    if (u >= g.H) u -= g.H;
    const int y = a < eh ? b * g.H + u : g.B * g.H, c0 = 32 * s;
    if (wc == c.seam) {
        const int n = c.n1 - c0;                          // slots of the strip in front of the seam
        if (n >= 32) {
            tc::tma_load_4d(dst, &m.seam_fa, ch, c0, 0, y, bar);
        } else if (n <= 0) {
            tc::tma_load_4d(dst, &m.seam_fb, ch, -n, 0, y, bar);
        } else {
            tc::tma_load_4d(dst, &m.seam_a, ch, c0, 0, y, bar);
            if (n + c.skip < 32) tc::tma_load_4d(dst + (n + c.skip) * ROWB, &m.seam_b, ch, c.skip, 0, y, bar);
        }
    } else if (wc == c.last) {
        tc::tma_load_4d(dst, &m.last, ch, c0, 0, y, bar);
    } else if (wc >= c.first_wrapped) {
        tc::tma_load_4d(dst, &m.wrapped, ch, c0, wc - c.first_wrapped, y, bar);
    } else {
        tc::tma_load_4d(dst, &m.row, ch, c0, wc, y, bar);
    }
}

// A window whose rows from `ha` on carry another mask label than those before is two windows where a 128-slot tile ends between them: the
// tiles of one part see none of the other's.  The first part's tiles, 0 where the window is one.  `row_slots`: slots of a window row.
__host__ __device__ __forceinline__ int part_tiles(int ha, int eh, int row_slots) { return ha > 0 && ha < eh && ha * row_slots % 128 == 0 ? ha * row_slots / 128 : 0; }

// Gangs of the one-pass backward (attn_bwd_onepass.cu), whose CTAs share the key tiles of a window (or of a part of one), `tiles` of them.
// The first tile that CTA `member` takes, where `seq` tiles were dealt before; then every gang-th.
__host__ __device__ __forceinline__ int gang_first_tile(int member, int seq, int gang) { return (member + gang - seq % gang) % gang; }
// The chunk of queries that tile `kt` starts at.
__host__ __device__ __forceinline__ int gang_first_chunk(int kt, int tiles, int gang, bool rotate) {
    const int ranks = gang < tiles ? gang : tiles;
    return rotate ? kt % ranks * tiles / ranks : 0;
}
// A tile's place in the order of those that add to chunk c: the tiles' own, or (rotate) from round to round of the gang's CTAs and in
// each from the one that starts at the chunk, or last in front of it, downwards.
__host__ __device__ __forceinline__ int gang_place(int kt, int c, int tiles, int gang, bool rotate) {
    if (!rotate) return kt;
    const int n = gang < tiles ? gang : tiles, j = kt % n, round = kt - j, in_round = n < tiles - round ? n : tiles - round;
    const int last = ((c + 1) * n - 1) / tiles, r = (last < in_round - 1 ? last : in_round - 1) - j;
    return round + (r < 0 ? r + in_round : r);
}

// slot (a, b) of a window -> grid token
__device__ __forceinline__ int win_token(const Geo& g, int wr, int wc, int a, int b) {
    int u = wr * g.w + a + g.sh;
    if (u >= g.H) u -= g.H;
    int v = wc * g.w + b + g.sw;
    if (v >= g.W) v -= g.W;
    return u * g.W + v;
}

}  // namespace terra
