// Window rows by tiled bulk copies (TMA), shared by the large-window tcgen05 kernels.
//
// On a grid of complete windows whose longitude shift is a multiple of 8, the tokens of one window row are one run of
// consecutive tokens of the tensor, or two where the rolled row crosses the longitude seam, each a multiple of 8 long.
// A tensor is described as [tokens, heads * d] with boxes of 32 columns (one 64-byte-swizzled part of a row) by 128,
// 64, 32, 16 or 8 tokens; a run is covered by the largest boxes that fit (the copy engine's time per box grows far
// slower than the box: 2 KB boxes reach a third of the bytes per clock of 8 KB boxes).
#pragma once
#include <cuda.h>

#include "swin_common.cuh"
#include "tc_common.cuh"

namespace terra {

struct RowMaps3 {
    // boxes of 32, 16, 8, 64 and 128 tokens x one part of a row: 32 columns (64-byte swizzle) or 64 columns (128-byte swizzle)
    CUtensorMap m[5];
};

// host: the maps of one tensor (`token_stride` in elements, parts of `part_cols` columns); false if the driver's encoder is not available
bool make_row_maps3(RowMaps3* maps, const Geo& g, const void* base, int token_stride, int part_cols);

// host: the geometry the bulk-copy loaders are written for
inline bool bulk_rows_shape(const Geo& g) {
    return (g.w == 64 || g.w == 128) && g.H % g.w == 0 && g.W % g.w == 0 && g.sw % 8 == 0 &&
           (long long)g.B * g.H * g.W < 0x7fffffffLL;
}

// device (ROWB = bytes of a part's row: 64 or 128): the copies of `n_run` slots (a multiple of 8) of window row `a`, from window column `b0` (a multiple of 8) on,
// of window row-index `wr` in sample `b`: ROWB bytes per slot from `dst` on (a multiple of 8 rows into a swizzled
// region), columns from xc on of every token; `v0` = the window's first token column after the roll.  The bytes
// are counted on `bar`.
template <int ROWB>
__device__ __forceinline__ void bulk_copy_window_run(const RowMaps3& m3, uint32_t dst, const Geo& g, int b, int wr, int v0, int a,
                                                     int b0, int n_run, int xc, uint32_t bar) {
    int u = wr * g.w + a + g.sh;
    if (u >= g.H) u -= g.H;
    const int y0 = (b * g.H + u) * g.W;
    int vs = v0 + b0;
    if (vs >= g.W) vs -= g.W;
    const int n1 = min(n_run, g.W - vs);          // tokens up to the seam; the rest starts at column 0
    int y = y0 + vs, n = n1;
#pragma unroll
    for (int seg = 0; seg < 2; ++seg) {
        while (n >= 128) { tc::tma_load_2d(dst, &m3.m[4], xc, y, bar); dst += 128 * ROWB; y += 128; n -= 128; }
        if (n >= 64) { tc::tma_load_2d(dst, &m3.m[3], xc, y, bar); dst += 64 * ROWB; y += 64; n -= 64; }
        while (n >= 32) { tc::tma_load_2d(dst, &m3.m[0], xc, y, bar); dst += 32 * ROWB; y += 32; n -= 32; }
        if (n >= 16) { tc::tma_load_2d(dst, &m3.m[1], xc, y, bar); dst += 16 * ROWB; y += 16; n -= 16; }
        if (n >= 8) { tc::tma_load_2d(dst, &m3.m[2], xc, y, bar); dst += 8 * ROWB; }
        y = y0;
        n = n_run - n1;
    }
}
// the whole window row
template <int ROWB>
__device__ __forceinline__ void bulk_copy_window_row(const RowMaps3& m3, uint32_t dst, const Geo& g, int b, int wr, int v0, int a,
                                                     int xc, uint32_t bar) {
    bulk_copy_window_run<ROWB>(m3, dst, g, b, wr, v0, a, 0, g.w, xc, bar);
}

}  // namespace terra
