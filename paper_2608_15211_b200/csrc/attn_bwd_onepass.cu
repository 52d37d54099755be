// One-pass backward on the tcgen05 tensor cores for window sides 9 .. 128 at head dim 128, 11 .. 128 at 64 and 17 .. 128 at 32, any grid:
// P and dS of a (window, head) are computed once and feed dQ, dK, dV and dBias.
//
// A persistent CTA takes (batch, window, head) units.  Per 128-key tile of a window it keeps K and V in shared memory and
// streams Q and dO in half chunks of 64 query slots (slots: win_tiles.cuh).  TMEM lanes = keys, columns = queries:
//   S^T = K Q^T, dP^T = V dO^T                                    (SS MMAs, N = 64)
//   P^T = exp2(S^T scale + bias - lse), dS^T = P^T (dP^T - delta)   (eight elementwise warps, in TMEM and shared memory)
//   dV += P^T dO, dK += dS^T Q                                    (A from TMEM)
//   dQ  += dS K     head dims 32, 64: per 128 queries, A = dS^T from shared memory read transposed
//   dQ^T = K^T dS^T  head dim 128: per half chunk, over the dP^T columns of its own buffer (TMEM has no others left)
// dQ sums over the window's key tiles: in TMEM where it fits (head dim 32, windows of at most 256 slots), else in a slab of
// fp32 that belongs to the CTA (one thread adds to one address, in key-tile order, so the sum has a fixed order).  Few
// (window, head) units: a window's key tiles are split over 2, 4 or 8 CTAs with a slab each.
// Sides above 32 (ST): window rows in strips of 32 slots (win_tiles.cuh), a strip taking the place of a row; bias and statistics from L2; gangs of
// CTAs share a window (Params).  Of a window whose mask label changes between two tiles each part is a window (part_tiles).
//
// The elementwise warps read and write TMEM in the fragment layout of mma.m16n8 (tcgen05.ld.16x256b): a thread holds 4 key
// rows x 8 query columns of every 32 x 32 block, at key offsets g + 8 m and query offsets 8 k + 2 t + e (g = lane / 4,
// t = lane % 4).  All (k, m) with one difference k - m share one bias entry and one bias-gradient entry, so a thread reads
// 14 bias values for 32 pairs and folds 32 dS values into 14 sums in registers; with one row per thread each pair costs a
// shared-memory load for the bias and a load and a store (or a shuffle, or an atomic) for its gradient.
// Measured, this kernel and what it needs around it against the kernels it replaces (dK / dV and dQ / dBias kernels that both
// recomputed P and dS; the latter on mma.sync wherever a window was not a complete 32 x 32 one): 256 x 512 tokens, 12 x 64,
// 32 x 32 windows 3.0 -> 2.1 ms; 255 x 540, the same 8.8 -> 2.2 ms; 288 x 544, 8 x 128, 16 x 16 windows 3.6 -> 1.1 ms; 64 x 128,
// 32 x 32 windows 32.2 -> 23.2 ms; 256 x 640, 8 x 128, 128 x 128 windows 51 -> 32 ms; 111 x 398, 12 x 128, side 64 25.4 -> 4.2 ms.  It is bound by the elementwise warps' chain per half chunk (issue slots 36 %, tensor pipe 26 %, DRAM 14 %),
// at head dim 128 with 32 x 32 windows by L2: 148 windows in flight restream their Q and dO and hold their dQ slabs, 1 MB each; on 96 x
// 160 tokens 7.3 GB are read and 4.0 GB written for 0.9 GB of tensors, and 15 % of L2's sector reads hit.
// dS^T leaves for shared memory by stmatrix in the layout the dQ product reads.
//
// Roles (512 threads): warps 0-3 / 4-7 elementwise on the even / odd half chunks, warps 8-11 read accumulators out of
// TMEM (dQ, dK, dV), warp 12 issues the products (dV, dK, dQ), warp 14 the scores (S^T, dP^T), warp 13 every copy, warp 15
// walks over the units, hands the others a descriptor per key tile and copies the tables.  Half chunks are numbered through the CTA's run and
// use TMEM buffer (number mod 2).  Shared-memory slots for K, V and query half chunks come from one pool in FIFO order, so
// the next tile's K and V are on their way while the current tile's last half chunks are worked on.
// Every mbarrier wait is bounded; on expiry the CTA raises an abort flag, all roles leave their loops, TMEM is
// released and the host reads the device status word.
#include "swin_common.cuh"
#include "swin_kernels.h"
#include "tc_common.cuh"
#include "win_tiles.cuh"

#include <cmath>
#include <cstring>

// fp16 build of this file (through the _f16 wrapper file): names of its own
#ifdef TERRA_ELEM_F16
#define g_bwd_onepass_timeout g_bwd_onepass_timeout_f16
#define launch_bwd_onepass launch_bwd_onepass_f16
#define read_bwd_onepass_status read_bwd_onepass_status_f16
#endif

namespace terra {

__device__ int g_bwd_onepass_timeout = 0;   // set when a bounded wait expired in any CTA of the kernel below

namespace {

using namespace tc;

constexpr int kThreads = 512;
constexpr int kWorkWarps = 8, kReadWarp0 = 8, kProductWarp = 12, kLoaderWarp = 13, kScoreWarp = 14, kPlanWarp = 15;
// Registers a thread: at launch, then of the elementwise, read-out and other warps.  The read-out's 64 accumulator values and addresses
// need 120 at head dims 64 and 128 and with strips (with 104 it spilled: 111 x 398 tokens, 12 x 128, side 64 5.1 ms, so 4.3; 288 x 544, 8 x 128, side 16 950 us, so 914).
// At head dim 32 the elementwise warps keep them (2 x 256 x 544, 13 heads, side 32: 3085 -> 3033).
constexpr int kRegsLaunch = 128, kRegsOther = 72;
template <int D, bool ST>
struct Regs {
    static constexpr int kWork = D == 32 && !ST ? 168 : 160, kRead = D == 32 && !ST ? 104 : 120;
    static_assert(2 * kWork + kRead + kRegsOther <= 4 * kRegsLaunch, "register hand-over does not balance");
    static_assert(kWork >= kRegsLaunch && kRead <= kRegsLaunch && kRegsOther <= kRegsLaunch, "only the elementwise warps take registers");
};
constexpr int kTile = 128, kHalf = 64;
constexpr int kDescs = 8;                                                             // ring of tile descriptors
constexpr int kScrLine = 160;                                                         // see flush_sums

template <int D, int RW, bool ST = false>
struct Lay {
    static constexpr int kParts = D == 128 ? 2 : 1, kRowB = D >= 64 ? 128 : 64;      // channel parts of a row, bytes of a part's row
    static constexpr int kPartCh = kRowB / 2;
    static constexpr int kSlotB = kTile * D * 2;                                      // K tile, V tile, or Q and dO of a half chunk
    // at least 6: the first half chunk of the next tile is loaded before the current tile's last one is done with
    static constexpr int kSlots = D == 128 ? 6 : D == 64 ? 8 : 14;
    static constexpr int kDsTiles = D == 128 ? 2 : 4, kDsB = kTile * kHalf * 2;       // dS^T tiles: 128 keys x 64 queries
    static constexpr int kOffDs = kSlots * kSlotB, kOffScr = kOffDs + kDsTiles * kDsB;
    static constexpr int kScrB = D == 128 ? 0 : 2 * 8 * kScrLine;                     // per elementwise warp: see flush_sums
    // per half chunk (ring of kTabs): 64 queries' statistics, then the bias rows its pieces meet, twice (the second copy shifted
    // by one entry and 16 banks away, so that lanes with even and odd g read different banks); head dim 128 has no room
    // and reads them from global memory
    // windows that are two parts (see part_tiles) as such; at head dim 32 what it takes costs all windows 5 % (2 x 256 x 544, 13 x 32, side 32)
    static constexpr bool kTwo = ST || D != 32;
    static constexpr bool kTables = D != 128 && !ST, kGang = ST;
    static constexpr int kTabs = 4, kBiasRows = kTile / RW + kHalf / RW - 1, kCopyB = kBiasRows * 2 * RW * 4;
    static constexpr int kOffCopy0 = 512, kOffCopy1 = 512 + (kCopyB + 127) / 128 * 128 + 64;
    static constexpr int kTabB = kTables ? (kOffCopy1 + kCopyB + 127) / 128 * 128 : 0;
    static constexpr int kOffTab = kOffScr + kWorkWarps * kScrB;
    static constexpr int kOffDesc = kOffTab + kTabs * kTabB;
    static constexpr int kOffBars = kOffDesc + kDescs * 64;
    static constexpr int kSmemBytes = kOffBars + 640;
    static_assert(kSmemBytes <= 232448, "shared memory of one CTA");
    // TMEM columns.  Buffer b: S^T at 128 b, dP^T at 128 b + 64.  Head dims 32 and 64: P^T and dS^T (packed) have places of
    // their own, so that the next scores are computed while the products read them; at head dim 128 they lie over
    // S^T and dP^T.
    static constexpr bool kOwnP = D != 128;
    static constexpr int kColP = kOwnP ? 256 : 0, kStrideP = kOwnP ? 64 : 128, kDsOff = kOwnP ? 32 : 64;   // P^T of buffer b; dS^T behind it
    static constexpr int kPieceP = kOwnP ? 16 : 32;                                   // from one piece's 16 packed columns to the next's
    static constexpr int kColAcc = kOwnP ? 384 : 256;                                 // dV, dK
    // dQ: head dim 32 two regions of its own; head dim 64 over P^T and dS^T of buffer 1 (per 128 queries); head dim 128
    // over dP^T of its buffer (per half chunk)
    static constexpr int kColDq = D == 32 ? 448 : D == 64 ? 320 : 64, kStrideDq = D == 32 ? 32 : 128;
    static constexpr int kResident = D == 32 && !ST ? 2 : 0;                                 // windows of that many 128-query chunks keep dQ in TMEM
};

template <bool ST>
using Maps = std::conditional_t<ST, WinStripMaps, WinMaps>;

// barriers (8 bytes each)
constexpr int kBFull = 0, kBEmpty = 16, kBSdp = 32, kBSFree = 34, kBDs = 36, kBPFree = 38, kBDq = 40, kBDqFree = 42, kBAcc = 44, kBAccFree = 45,
              kBDesc = 46, kBDescFree = kBDesc + kDescs, kBTab = kBDescFree + kDescs, kBTabFree = kBTab + 4, kBCount = kBTabFree + 4;

struct Params {
    Geo g;
    WinCols cols;
    int split_log2;                  // key tiles of a window are shared by 1 << split_log2 units
    int npad;                        // slots of a full window, rounded up to 128
    int rmax;                        // window rows rounded up to whole key tiles: bias-table rows run from -rmax to rmax - 1
    int rl;                          // floats of a bias-table row: 2 RW (ST: 64 for every strip of a full window row)
    // The launch's units: first those of the windows (row >= row1, any column), then of (row < row1, column >= col1); a launch of
    // the inner windows has the units of (row < row1, column < col1).
    int row1, col1, inner;
    int part_row, part_ha;           // the window row whose windows may be two parts, -1: none (see part_tiles), and the second part's first row
    int slab0;                       // first slab of the launch (two launches may overlap)
    int overlap;                     // the launch runs beside the one before it, which started when its prerequisites were complete
    // Gangs: `gang` CTAs work on the key tiles of one (window, head) after the other, each on every gang-th of the gang's tiles, and add
    // to the window's dQ slab in the tiles' order.  flags[slab][event][read-out warp] = number of the next tile that may add
    // (tiles numbered through the gang's run), flags[slab][events] = windows that are done with the slab.
    // Where every gang has one window only, the CTAs start at different chunks of its queries (`rotate`) instead of after one another.
    int gangs, gang, ring, events, rotate;
    int turn_log2;                   // dQ events that the CTAs take turns by
    unsigned* flags;
    long long units;
    const float4* rowstat;           // per (b, window, head) and slot pair: (-lse log2 e) x 2, delta x 2
    const float* bias0;              // [head][2 rmax][rl]: bias log2 e at (da + rmax, db + rl / 2), 0 outside the table
    const float* bias1;              // the same, shifted by one entry
    float* dbias_acc;                // [head][2 rmax][rl]
    const __nv_bfloat16 *q, *k, *v, *d_o;
    float4* slabs;                   // dQ partial sums: one slab of npad x D floats per CTA (per unit where windows are split)
};

// The pool's FIFO of shared-memory slots (4 bits each).  Loader and issuers step through the same sequence of loads and
// hold the same queue: a query half chunk's slot goes to the back when it is taken (slots are released in the order they
// were taken within a tile), a tile's V and K slots behind the tile's last half chunk.
template <int N>
struct SlotQueue {
    uint64_t q;
    __device__ __forceinline__ void init() {
        q = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) q |= (uint64_t)i << (4 * i);
    }
    __device__ __forceinline__ int pop() { const int s = (int)(q & 15); q >>= 4; return s; }
    __device__ __forceinline__ int take_half() { const int s = pop(); q |= (uint64_t)s << (4 * (N - 3)); return s; }
    __device__ __forceinline__ void end_tile(int sk, int sv) { q |= ((uint64_t)sv << (4 * (N - 2))) | ((uint64_t)sk << (4 * (N - 1))); }
};

// A key tile of a unit, as the planning warp hands it to the other roles.
struct TileDesc {
    int head, b, wr, wc;
    int eh, ew, kt;
    int nch, q0;           // chunks of 128 queries that the tile meets, and the first of them (see part_tiles)
    int ha, hb;            // window rows >= ha / columns >= hb carry the other shift-mask label (far outside: none do)
    int flags;             // 1: a tile (0: the end), 2: the unit's first, 4: its last
    int slab;
    int ns;                // ST: strips of a window row
    int seq, use, c0;      // gangs: number of the window's first tile, windows before on this slab; first chunk of queries
};

__device__ __forceinline__ float2 lds_f2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ float4 lds_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ float lds_f1(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts_f2(uint32_t addr, float2 v) {
    asm volatile("st.shared.v2.f32 [%0], {%1,%2};\n" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void red_f1(float* p, float v) { asm volatile("red.global.add.f32 [%0], %1;\n" ::"l"(p), "f"(v) : "memory"); }
__device__ __forceinline__ void red_f4(float4* p, float4 v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1,%2,%3,%4};\n" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// What an elementwise thread reads for 32 query columns: the bias pairs of its diagonals and the statistics of its columns.
// RW = 32: the piece is one window row of queries, the warp's keys one window row: diagonals 8 s + 2 t + e - g, s = -3 .. 3.
// RW = 16: two window rows of queries and of keys: three row differences d = -1, 0, 1, diagonals s = -1, 0, 1 each.
template <int RW>
struct Piece {
    static constexpr int kSums = RW == 32 ? 7 : 9;
    // which of them pair (k, m) belongs to
    __host__ __device__ static constexpr int sum_of(int k, int m) { return RW == 32 ? k - m + 3 : ((k >> 1) - (m >> 1) + 1) * 3 + (k & 1) - (m & 1) + 1; }
    float2 bias[kSums];
    float4 st[4];                 // per k: (-lse log2 e) of columns 8 k + 2 t, + 1, then their deltas
    // `bp`: the thread's entry of row difference 0 of the piece and diagonal s = 0
    __device__ __forceinline__ void load(const float* __restrict__ bp, const float4* __restrict__ sp) {
#pragma unroll
        for (int i = 0; i < kSums; ++i) {
            const int off = RW == 32 ? 8 * (i - 3) : (i / 3 - 1) * 2 * RW + 8 * (i % 3 - 1);
            bias[i] = __ldg(reinterpret_cast<const float2*>(bp + off));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) st[k] = __ldg(sp + 4 * k);
    }
    // the same from shared memory
    __device__ __forceinline__ void load(uint32_t bp, uint32_t sp) {
#pragma unroll
        for (int i = 0; i < kSums; ++i) {
            const int off = RW == 32 ? 8 * (i - 3) : (i / 3 - 1) * 2 * RW + 8 * (i % 3 - 1);
            bias[i] = lds_f2(bp + 4 * off);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) st[k] = lds_f4(sp + 64 * k);
    }
};

// 32 accumulator columns of one row, scaled, as 64 bytes of 16-bit elements
__device__ __forceinline__ void store_scaled32(uint4* dst, const uint32_t (&r)[32], float f) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint4 a;
        a.x = pack_elem(__uint_as_float(r[c * 8 + 0]) * f, __uint_as_float(r[c * 8 + 1]) * f);
        a.y = pack_elem(__uint_as_float(r[c * 8 + 2]) * f, __uint_as_float(r[c * 8 + 3]) * f);
        a.z = pack_elem(__uint_as_float(r[c * 8 + 4]) * f, __uint_as_float(r[c * 8 + 5]) * f);
        a.w = pack_elem(__uint_as_float(r[c * 8 + 6]) * f, __uint_as_float(r[c * 8 + 7]) * f);
        dst[c] = a;
    }
}

// 32 accumulator columns of a row a lane, scaled, as 64 bytes of 16-bit elements of each row; four lanes exchange 16-byte pieces, so that they write
// the 64 bytes of one row after the other side by side.  Head dim 32, windows without a mask (2 x 256 x 544 tokens, 13 heads, side 32: 3250 -> 3056
// us); not faster elsewhere (masked, side 24: 1050 -> 1100; head dims 64, 128 at side 32 level, at side 16 6 % slower).  `off`: the lane's row in `base`, in elements (negative: none).
__device__ __forceinline__ void store_rows32(__nv_bfloat16* base, long long off, const uint32_t (&r)[32], float f, int lane) {
    uint32_t c[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) c[j][i] = pack_elem(__uint_as_float(r[8 * j + 2 * i]) * f, __uint_as_float(r[8 * j + 2 * i + 1]) * f);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const bool up = lane & (1 << s);
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const int lo = s ? p : 2 * p, hi = s ? p + 2 : 2 * p + 1;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t x = __shfl_xor_sync(0xffffffffu, up ? c[lo][i] : c[hi][i], 1 << s);
                if (up) c[lo][i] = x; else c[hi][i] = x;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long at = __shfl_sync(0xffffffffu, off, (lane & ~3) + i);
        if (at >= 0) reinterpret_cast<uint4*>(base + at)[lane & 3] = make_uint4(c[i][0], c[i][1], c[i][2], c[i][3]);
    }
}

// One step (32 keys x 16 queries, columns k = 2 U and 2 U + 1 of the piece): P = exp2(S scale + bias - lse), dS = P (dP - delta);
// packed P and dS go to TMEM, dS also to its shared-memory tile, and the piece's sums per diagonal grow.
// MASK: bit 2 k + e of ok[m] allows the pair.
template <int RW, int MASK, int U>
__device__ __forceinline__ void step_math(const uint32_t (&rs)[2][8], const uint32_t (&rp)[2][8], uint32_t t_p, uint32_t t_ds, uint32_t st_addr,
                                          const Piece<RW>& pc, const uint32_t (&ok)[4], float scale, float2 (&sum)[Piece<RW>::kSums]) {
    uint32_t pp[2][4], pd[2][4];                  // [m / 2][2 (k - 2 U) + m % 2]
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int k = 2 * U + kk, hl = m >> 1, mi = m & 1, i = Piece<RW>::sum_of(k, m);
            float x0, x1, t0, t1, d0, d1;
            fma2(x0, x1, __uint_as_float(rs[hl][4 * kk + 2 * mi]), __uint_as_float(rs[hl][4 * kk + 2 * mi + 1]), scale, pc.bias[i].x, pc.bias[i].y);
            add2vv(x0, x1, x0, x1, pc.st[k].x, pc.st[k].y);
            if (MASK) {
                x0 = (ok[m] & (1u << (2 * k))) ? x0 : -INFINITY;
                x1 = (ok[m] & (2u << (2 * k))) ? x1 : -INFINITY;
            }
            const float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
            sub2(t0, t1, __uint_as_float(rp[hl][4 * kk + 2 * mi]), __uint_as_float(rp[hl][4 * kk + 2 * mi + 1]), pc.st[k].z, pc.st[k].w);
            mul2(d0, d1, p0, p1, t0, t1);
            add2vv(sum[i].x, sum[i].y, sum[i].x, sum[i].y, d0, d1);
            pp[hl][2 * kk + mi] = pack_elem(p0, p1);
            pd[hl][2 * kk + mi] = pack_elem(d0, d1);
        }
    }
#pragma unroll
    for (int hl = 0; hl < 2; ++hl) {
        tmem_st_frag8(t_p + 8 * U + ((uint32_t)(16 * hl) << 16), pp[hl]);
        tmem_st_frag8(t_ds + 8 * U + ((uint32_t)(16 * hl) << 16), pd[hl]);
        // matrices (m, k) = (2 hl, 2 U), (2 hl, 2 U + 1), (2 hl + 1, 2 U), (2 hl + 1, 2 U + 1)
        stmatrix_x4((st_addr ^ (32u * U)) + hl * 2048, pd[hl][0], pd[hl][2], pd[hl][1], pd[hl][3]);
    }
}

// The sums of both pieces of a half chunk -> one value per diagonal -> the head's bias-gradient table.  Thread (g, t) holds the
// part of diagonal 8 s + 2 t + e - g; diagonal d collects, for every g, the entry with 8 s + (2 t + e) = d + g.  The sums pass
// through shared memory: a line of five groups of 8 floats per g, group = s in order, so that lane l's entry of line g lies at
// l + 1 + g: one address and immediate offsets, and (lines 40 floats apart) no bank conflicts in either direction.  RW = 32:
// s = -3 .. 0 behind a group of zeros give diagonals l - 31, s = 0 .. 3 in front of one give l + 1; RW = 16: a round per row
// difference, s = -1 .. 1 between two groups of zeros, diagonals l - 15.  `acc`: where piece 0's diagonal -RW would go,
// `acc_row`: floats from there to piece 1's.
template <int RW>
__device__ __forceinline__ void flush_sums(uint32_t scr, const float2 (&sum)[2][Piece<RW>::kSums], int lane, float* acc, int acc_row) {
    constexpr int kRounds = RW == 32 ? 2 : 3;
    const uint32_t w = scr + (lane >> 2) * kScrLine + (lane & 3) * 8, rd = scr + (lane + 1) * 4;
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint32_t wj = w + j * 8 * kScrLine;
            if (RW == 32) {
                sts_f2(wj + (r ? 4 : 0) * 32, make_float2(0.f, 0.f));
#pragma unroll
                for (int i = 0; i < 4; ++i) sts_f2(wj + (r ? i : i + 1) * 32, sum[j][3 * r + i]);
            } else {
                if (r == 0) {
                    sts_f2(wj, make_float2(0.f, 0.f));
                    sts_f2(wj + 4 * 32, make_float2(0.f, 0.f));
                }
#pragma unroll
                for (int i = 0; i < 3; ++i) sts_f2(wj + (i + 1) * 32, sum[j][3 * r + i]);
            }
        }
        __syncwarp();
        float v[2][8];
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int gg = 0; gg < 8; ++gg) v[j][gg] = lds_f1(rd + j * 8 * kScrLine + gg * (kScrLine + 4));
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float x = ((v[j][0] + v[j][1]) + (v[j][2] + v[j][3])) + ((v[j][4] + v[j][5]) + (v[j][6] + v[j][7]));
            float* dst = acc + j * acc_row + (RW == 32 ? (r ? 33 : 1) : (r - 1) * 2 * RW + 1) + lane;
            if ((RW == 32 && r == 0) || lane < 31) red_f1(dst, x);
        }
    }
}

// One half chunk of a warp (32 keys x 64 queries): scores in TMEM to P and dS in their places, in four steps of 16 queries.
// `t_s`: S^T (dP^T 64 columns behind it); `t_p`: P^T (dS^T kDsOff behind it).  Head dims 32 and 64: the next step's scores are
// loaded ahead, pc[0] holds the first piece's tables and the second's follow from shared memory (`tab_b`, `tab_s`).  Head dim
// 128: pc holds both pieces' tables, whose trip to L2 is the longer one.
template <int D, int RW, int MASK, bool ST>
__device__ __forceinline__ void half_chunk(uint32_t t_s, uint32_t t_p, uint32_t st_addr, Piece<RW> (&pc)[2], uint32_t tab_b, uint32_t tab_s,
                                           const uint32_t (&okm)[2][4], float scale, float2 (&sum)[2][Piece<RW>::kSums], int lane, uint32_t bar_sfree) {
    using L = Lay<D, RW, ST>;
    constexpr int kAhead = L::kTables ? 1 : 0;
    uint32_t rs[1 + kAhead][2][8], rp[1 + kAhead][2][8];
    auto ld = [&](int i) {
#pragma unroll
        for (int hl = 0; hl < 2; ++hl) {
            tmem_ld_frag16(t_s + 16 * i + ((uint32_t)(16 * hl) << 16), rs[i & kAhead][hl]);
            tmem_ld_frag16(t_s + 64 + 16 * i + ((uint32_t)(16 * hl) << 16), rp[i & kAhead][hl]);
        }
    };
    ld(0);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int j = i >> 1;
        if ((i & 1) == 0) {
#pragma unroll
            for (int x = 0; x < Piece<RW>::kSums; ++x) sum[j][x] = make_float2(0.f, 0.f);
        }
        if (!kAhead && i > 0) ld(i);
        tmem_ld_wait();
        if (kAhead && i < 3) ld(i + 1);
        if (L::kOwnP && i == 3) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_sfree);
        }
        const uint32_t tp = t_p + L::kPieceP * j, sa = st_addr ^ (64u * j);
        const Piece<RW>& pj = pc[L::kTables ? 0 : j];
        if ((i & 1) == 0) step_math<RW, MASK, 0>(rs[i & kAhead], rp[i & kAhead], tp, tp + L::kDsOff, sa, pj, okm[j], scale, sum[j]);
        else step_math<RW, MASK, 1>(rs[i & kAhead], rp[i & kAhead], tp, tp + L::kDsOff, sa, pj, okm[j], scale, sum[j]);
        // the second piece: 32 / RW row differences further
        if (L::kTables && i == 1) pc[0].load(tab_b + (32 / RW) * 2 * RW * 4, tab_s + 256);
    }
}

// KIND 0: windows whose slots all hold tokens and whose tokens share one mask label.  1: windows that need the mask.  2: both (head
// dim 128).  Two launches instead of a branch: with both bodies in one kernel the unmasked one ran 1.14 times as long (the
// elementwise warps are sensitive to what the compiler and the instruction caches make of them), at head dim 128 it is not
// what bounds the kernel.
template <int D, int RW, int KIND, bool ST>
__global__ void __launch_bounds__(kThreads, 1)
swin_bwd_onepass_kernel(const __grid_constant__ Params p, __nv_bfloat16* __restrict__ dq, __nv_bfloat16* __restrict__ dk,
                        __nv_bfloat16* __restrict__ dv, const __grid_constant__ Maps<ST> mq, const __grid_constant__ Maps<ST> mk,
                        const __grid_constant__ Maps<ST> mv, const __grid_constant__ Maps<ST> mg) {
    using L = Lay<D, RW, ST>;
    constexpr int kParts = L::kParts, kRowB = L::kRowB, kG = kHalf / RW;
    constexpr bool kExchange = D == 32 && KIND == 0;
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t smem0 = smem_u32(smem), bar0 = smem0 + L::kOffBars;
    auto bar = [&](int i) { return bar0 + 8u * i; };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kOffBars + 8 * kBCount);
    volatile int* cta_abort = reinterpret_cast<volatile int*>(smem + L::kOffBars + 8 * kBCount + 8);
    const Geo& g = p.g;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid == 0) {
        for (int s = 0; s < L::kSlots; ++s) {
            mbar_init(bar(kBFull + s), 1);
            mbar_init(bar(kBEmpty + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(kBSdp + b), 1);          // S^T, dP^T of a half chunk are in buffer b (and its P^T, dS^T places are free)
            mbar_init(bar(kBSFree + b), 4);        // ... and read by the elementwise warps (head dims 32, 64)
            mbar_init(bar(kBDs + b), 4);           // P^T, dS^T are in their place
            mbar_init(bar(kBPFree + b), 1);        // ... and read by the products
            mbar_init(bar(kBDq + b), 1);           // dQ region b is final (for this key tile, or the window)
            mbar_init(bar(kBDqFree + b), 4);       // ... and read
        }
        mbar_init(bar(kBAcc), 1);                  // dV, dK of a key tile are final
        mbar_init(bar(kBAccFree), 4);              // ... and read
        for (int i = 0; i < kDescs; ++i) {
            mbar_init(bar(kBDesc + i), 1);
            mbar_init(bar(kBDescFree + i), kWorkWarps + 7);
        }
        for (int i = 0; i < L::kTabs; ++i) {
            mbar_init(bar(kBTab + i), 1);          // tables of a half chunk
            mbar_init(bar(kBTabFree + i), 4);
        }
        *cta_abort = 0;
        fence_barrier_init();
    }
    if (warp == kProductWarp) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // the next tile's descriptor; false at the end of the run (or after an expired wait)
    unsigned desc_n = 0;
    TileDesc td;
    auto next_tile = [&]() {
        const unsigned i = desc_n % kDescs;
        if (!mbar_wait_all(bar(kBDesc + i), (desc_n / kDescs) & 1, cta_abort)) return false;
        const int4* src = reinterpret_cast<const int4*>(smem + L::kOffDesc + i * 64);
        const int4 d0 = src[0], d1 = src[1], d2 = src[2];
        td.head = d0.x; td.b = d0.y; td.wr = d0.z; td.wc = d0.w;
        td.eh = d1.x; td.ew = d1.y; td.kt = d1.z; td.nch = L::kTwo ? d1.w & 0xffff : d1.w; td.q0 = L::kTwo ? d1.w >> 16 : 0;
        td.ha = d2.x; td.hb = d2.y; td.flags = d2.z; td.slab = d2.w;
        if (ST) {
            const int4 d3 = src[3];
            td.ns = d3.x; td.seq = d3.y; td.use = d3.z; td.c0 = d3.w;
        } else {
            td.ns = 1;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kBDescFree + i));
        ++desc_n;
        return (td.flags & 1) != 0;
    };

    // the launch of the masked windows may take the SMs that this one leaves (it waits for this one's end before its own)
    if (KIND == 0) let_dependents_start();

    if (warp < kWorkWarps) {
        // ------------------------------------------------------------------ elementwise: the half chunks of buffer b
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(Regs<D, ST>::kWork));
        const int b = warp >> 2, wq = warp & 3, gl = lane >> 2, t = lane & 3;
        const float scale = g.scale_log2e;
        const uint32_t tq = tmem + ((uint32_t)(32 * wq) << 16);
        const uint32_t t_s = tq + 128u * b, t_p = tq + L::kColP + L::kStrideP * b;
        const int rl = ST ? p.rl : 2 * RW, head_f = 2 * p.rmax * rl;
        // stmatrix: lane l addresses row l % 8 of the four matrices (m, k) = (l / 16, l / 8 % 2)
        const uint32_t st_off = (uint32_t)((32 * wq + 8 * (lane >> 4) + (lane & 7)) * 128 + ((((lane >> 3) & 1) ^ (lane & 7)) << 4));
        const uint32_t scr0 = D == 128 ? smem0 + L::kOffDs + b * L::kDsB + 32 * wq * 128 : smem0 + L::kOffScr + warp * L::kScrB;
        unsigned n = 0;                                      // half chunks of this buffer so far
        int a_k0, nh, left, ha, row0, hc = 0;
        int c_k0 = 0;                                        // ST: first column of the warp's keys
        bool masked;
        uint32_t rowbits, qbits, sp;
        const int lane_e = 2 * t - gl - (gl & 1) + (ST ? rl / 2 : RW);       // the thread's entry within a table row (even: both copies are read in pairs)
        const float* tbl = ((gl & 1) ? p.bias1 : p.bias0) + lane_e;
        // in a staged table: piece 0's row difference 0 is row 128 / RW - 1 - (the warp's first key row in the tile)
        const uint32_t tab_b0 = smem0 + L::kOffTab + ((gl & 1) ? L::kOffCopy1 : L::kOffCopy0) + ((kTile / RW - 1 - (RW == 32 ? wq : 2 * wq)) * 2 * RW + lane_e) * 4;
        const uint32_t tab_s0 = smem0 + L::kOffTab + t * 16;
        Piece<RW> pc[2];
        // the next tile: what its half chunks have in common
        auto enter_tile = [&]() {
            if (!next_tile()) return false;
            hc = 2 * td.q0 + (ST ? 2 * td.c0 + b : b);
            if (ST) left = td.nch;
            nh = 2 * (td.q0 + td.nch);
            ha = td.ha;
            a_k0 = td.kt * (kTile / RW) + (RW == 32 ? wq : 2 * wq);
            if (ST) {
                const int u = a_k0;
                a_k0 = unit_row(u, td.ns);
                c_k0 = 32 * (u - a_k0 * td.ns);
            }
            const bool labels = (ha > 0 && ha < td.eh && (!L::kTwo || part_tiles(ha, td.eh, td.ns * RW) == 0)) || (td.hb > 0 && td.hb < td.ew);
            masked = KIND == 1 || (KIND == 2 && (labels || td.ew < td.ns * RW || (td.kt + 1) * (kTile / RW) > td.eh * td.ns));
            rowbits = 0;                                     // bits m: the row holds a key; bits 4 + m: it lies behind hb
            qbits = 0;
            if (masked) {
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int a = a_k0 + (RW == 32 ? 0 : m >> 1), bb = c_k0 + gl + 8 * (RW == 32 ? m : m & 1);
                    rowbits |= (((a < td.eh && bb < td.ew) ? 1u : 0u) << m) | ((bb >= td.hb ? 16u : 0u) << m);
                    const int q0 = (RW == 32 ? 8 * m : 8 * (m & 1)) + 2 * t;
                    qbits |= ((q0 >= td.hb ? 1u : 0u) | (q0 + 1 >= td.hb ? 2u : 0u)) << (2 * m);
                }
            }
            // piece 0 of half chunk 0: row difference a_q - a_k = -a_k0
            row0 = td.head * head_f + (p.rmax - a_k0) * rl - c_k0;
            sp = (uint32_t)(((td.b * g.Mh + td.wr) * g.Mw + td.wc) * g.heads + td.head);
            return true;
        };
        auto bias_ptr = [&]() { return tbl + row0 + hc * kG * (2 * RW); };
        // ST: floats from row0 to piece j of half chunk hc
        auto piece_at = [&](int j) {
            const int u = 2 * hc + j, a = unit_row(u, td.ns);
            return a * rl + 32 * (u - a * td.ns);
        };
        auto stat_ptr = [&]() { return p.rowstat + (size_t)sp * (p.npad / 2) + (hc * 32 + t); };
        bool live = enter_tile();
        auto load_tables = [&]() {
            pc[0].load(ST ? tbl + row0 + piece_at(0) : bias_ptr(), stat_ptr());
            pc[1].load(ST ? tbl + row0 + piece_at(1) : bias_ptr() + (32 / RW) * 2 * RW, stat_ptr() + 16);
        };
        if (live && !L::kTables) load_tables();
        while (live) {
            float2 sum[2][Piece<RW>::kSums];
            const uint32_t st_addr = smem0 + L::kOffDs + (D == 128 ? (uint32_t)b : 2 * (n & 1) + b) * L::kDsB + st_off;
            const unsigned ti = (2 * n + b) % L::kTabs, tuse = (2 * n + b) / L::kTabs;
            const uint32_t tb = tab_b0 + ti * L::kTabB, ts = tab_s0 + ti * L::kTabB;
            if (L::kTables) {
                if (!mbar_wait_all(bar(kBTab + ti), tuse & 1, cta_abort)) break;
                pc[0].load(tb, ts);
            }
            if (!mbar_wait_all(bar(kBSdp + b), n & 1, cta_abort)) break;
            tc_fence_after();
            uint32_t okm[2][4] = {};
            if (!masked) {
                half_chunk<D, RW, KIND == 1 ? 1 : 0, ST>(t_s, t_p, st_addr, pc, tb, ts, okm, scale, sum, lane, bar(kBSFree + b));
            } else {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    int aq = hc * kG + j * (32 / RW);
                    if (ST) {
                        const int u = aq;
                        aq = unit_row(u, td.ns);
                        qbits = 0;
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const int q0 = 32 * (u - aq * td.ns) + 8 * m + 2 * t;
                            qbits |= ((q0 >= td.hb ? 1u : 0u) | (q0 + 1 >= td.hb ? 2u : 0u)) << (2 * m);
                        }
                    }
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const bool ka = a_k0 + (RW == 32 ? 0 : m >> 1) >= ha;
                        const uint32_t rows = RW == 32 ? (((aq >= ha) == ka) ? 0xffu : 0u)
                                                       : (((aq >= ha) == ka) ? 0x0fu : 0u) | (((aq + 1 >= ha) == ka) ? 0xf0u : 0u);
                        okm[j][m] = (rowbits & (1u << m)) ? ((rowbits & (16u << m)) ? qbits : ~qbits) & rows : 0u;
                    }
                }
                half_chunk<D, RW, KIND == 0 ? 0 : 1, ST>(t_s, t_p, st_addr, pc, tb, ts, okm, scale, sum, lane, bar(kBSFree + b));
            }
            fence_proxy_async();
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar(kBDs + b));
                if (L::kTables) mbar_arrive(bar(kBTabFree + ti));
            }
            // the next half chunk's tables are on their way while the rest is done
            float* acc = p.dbias_acc + row0 + (ST ? piece_at(0) + rl / 2 - 32 : hc * kG * (2 * RW));
            const int acc_row = ST ? piece_at(1) - piece_at(0) : (32 / RW) * 2 * RW;
            hc += 2;
            if (ST) {
                if (hc >= nh) hc -= 2 * td.nch;
                if (--left == 0) live = enter_tile();
            } else if (hc >= nh) {
                live = enter_tile();
            }
            if (live && !L::kTables) load_tables();
            // The bias gradient, while the products are computed.  Head dim 128 has no shared memory to spare: the sums go
            // through the warp's own rows of the dS^T tile once the dQ product has read them.
            if (D == 128 && !mbar_wait_all(bar(kBDq + b), n & 1, cta_abort)) break;
            flush_sums<RW>(scr0, sum, lane, acc, acc_row);
            if (D == 128) __syncwarp();
            ++n;
        }
    } else if (warp < kProductWarp) {
        // ------------------------------------------------------------------ read-out
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(Regs<D, ST>::kRead));
        const int wq = warp & 3, row = 32 * wq + lane;          // TMEM lane
        const uint32_t tl = tmem + ((uint32_t)(32 * wq) << 16);
        const float out_scale = g.scale_log2e * kLn2;
        const bool split = p.split_log2 > 0;
        unsigned n = 0, na = 0;                                  // dQ events, key tiles so far
        uint32_t dq_use = 0;
        bool ok = true;
        // 32 columns of this thread's row to the slab (as eight float4s 128 threads apart) and from it
        auto to_slab = [&](float4* s4, const uint32_t (&v)[32], bool add) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 x = make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]), __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3]));
                if (add) red_f4(s4 + i * 128, x);
                else __stcg(s4 + i * 128, x);
            }
        };
        auto from_slab = [&](const float4* s4, uint32_t (&v)[32]) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 o = __ldcg(s4 + i * 128);
                v[4 * i] = __float_as_uint(__uint_as_float(v[4 * i]) + o.x);
                v[4 * i + 1] = __float_as_uint(__uint_as_float(v[4 * i + 1]) + o.y);
                v[4 * i + 2] = __float_as_uint(__uint_as_float(v[4 * i + 2]) + o.z);
                v[4 * i + 3] = __float_as_uint(__uint_as_float(v[4 * i + 3]) + o.w);
            }
        };
        // Gangs.  A tile adds to a turn's part of its slab when the tile before it has, the window's first tile stores there when the slab's
        // last window is done with it.  This warp reads and writes the same rows of the slab in every CTA, so it only waits for its like.
        // The release in front of the signal waits for the adds to arrive; it is left until the next event, when most have.
        const bool ganged = L::kGang && p.gang > 1;
        auto flag = [&](int i) { return p.flags + ((size_t)td.slab * (p.events + 1) + i) * 4 + wq; };
        unsigned* pending = nullptr;
        unsigned pending_value = 0;
        auto place = [&](int c) { return gang_place(td.kt - td.q0, c, td.nch, p.gang, p.rotate); };
        auto signal = [&](unsigned* f, unsigned value) {
            __syncwarp();
            if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;\n" ::"l"(f), "r"(value) : "memory");
        };
        auto signal_pending = [&]() {
            if (pending) signal(pending, pending_value);
            pending = nullptr;
        };
        auto await_flag = [&](const unsigned* f, unsigned value) {
            const long long t0 = clock64();
            while (true) {
                unsigned v;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(f) : "memory");
                if (__all_sync(0xffffffffu, v >= value)) return true;
                if (__any_sync(0xffffffffu, *cta_abort != 0 || clock64() - t0 > 4000000000LL)) {
                    *cta_abort = 1;
                    return false;
                }
            }
        };
        // in front of event `ev` of a tile that is not a window's only one
        auto turn = [&](int ev, int at) {
            signal_pending();
            const bool starts = (ev & ((1 << p.turn_log2) - 1)) == 0;
            if (at == 0) return !starts || p.rotate || ev > 0 || await_flag(flag(p.events), td.use);
            return !starts || await_flag(flag(ev >> p.turn_log2), td.seq + at);
        };
        // behind it; `end`: the window's last
        auto turn_done = [&](int ev, int at, bool end) {
            if (end || ((ev + 1) & ((1 << p.turn_log2) - 1)) == 0) {
                pending = flag(ev >> p.turn_log2);
                pending_value = td.seq + at + 1;
            }
        };
        // the accumulator columns are handed back as soon as they are in registers: 64 at a time
        constexpr int kLd = D == 32 ? 1 : 2;
        auto hand_back = [&](int i) {
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(i));
        };
        while (ok && next_tile()) {
            bool first = td.flags & 2, last = td.flags & 4;
            const bool shared = ganged && td.nch > 1;
            int at = td.kt - td.q0;
            const size_t sample = (size_t)td.b * g.H * g.W;
            float4* slab = p.slabs + ((size_t)td.slab * p.npad + td.q0 * kTile) * (D / 4) + row;
            const int u0 = td.q0 * (kTile / RW);                 // the part's first window row (ST: strip)
            if (D == 128) {
                // dQ^T: lanes = channels, columns = the half chunk's queries
                for (int i = 0; i < 2 * td.nch; ++i, ++n) {
                    const int b = i & 1, rel = ST && i + 2 * td.c0 >= 2 * td.nch ? i + 2 * td.c0 - 2 * td.nch : ST ? i + 2 * td.c0 : i;
                    const int ev = ST && p.rotate ? 2 * td.q0 + rel : rel;       // (rotate: both parts of a window use one slab)
                    if (shared) {
                        if (p.rotate) {
                            at = place(rel >> 1);
                            first = at == 0;
                            last = at == td.nch - 1;
                        }
                        ok = turn(ev, at);
                    }
                    ok = ok && mbar_wait_all(bar(kBDq + b), (n >> 1) & 1, cta_abort);
                    if (!ok) break;
                    tc_fence_after();
                    uint32_t r[2][32];
                    tmem_ld32(tl + 128u * b + L::kColDq, r[0]);
                    tmem_ld32(tl + 128u * b + L::kColDq + 32, r[1]);
                    hand_back(kBDqFree + b);
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        float4* s4 = slab + (rel * 16 + hh * 8) * 128;
                        if (!last || split) {
                            to_slab(s4, r[hh], !first);
                        } else {
                            if (!first) from_slab(s4, r[hh]);
                            const int s0 = rel * kHalf + 32 * hh;
#pragma unroll
                            for (int jr = 0; jr < 32 / RW; ++jr) {
                                const int u = u0 + s0 / RW + jr, a = ST ? unit_row(u, td.ns) : u, c0 = ST ? 32 * (u - a * td.ns) : 0;
                                if (a >= td.eh) continue;
                                int v = td.wc * g.w + c0 + g.sw;
                                if (v >= g.W) v -= g.W;
                                __nv_bfloat16* base = dq + (sample + (size_t)win_token(g, td.wr, td.wc, a, c0) - v) * g.ts + td.head * D;
                                if (ST ? v + 32 <= g.W && c0 + 32 <= td.ew : v + td.ew <= g.W && td.ew == RW) {
                                    // two lanes exchange halves, so that each stores two channels of every other query
                                    uint32_t* d2 = reinterpret_cast<uint32_t*>(base + (size_t)(v + (row & 1)) * g.ts + (row & ~1));
#pragma unroll
                                    for (int i = 0; i < RW; i += 2) {
                                        const float x0 = __uint_as_float(r[hh][jr * RW + i]) * out_scale, x1 = __uint_as_float(r[hh][jr * RW + i + 1]) * out_scale;
                                        const float y = __shfl_xor_sync(0xffffffffu, (row & 1) ? x0 : x1, 1);
                                        *d2 = (row & 1) ? pack_elem(y, x1) : pack_elem(x0, y);
                                        d2 += g.ts;                       // two tokens of ts 16-bit elements
                                    }
                                } else {
#pragma unroll
                                    for (int i = 0; i < RW; ++i) {
                                        if (c0 + i < td.ew) {
                                            const uint32_t pkd = pack_elem(__uint_as_float(r[hh][jr * RW + i]) * out_scale, 0.f);
                                            *reinterpret_cast<uint16_t*>(base + (size_t)v * g.ts + row) = (uint16_t)pkd;
                                        }
                                        if (++v >= g.W) v = 0;
                                    }
                                }
                            }
                        }
                    }
                    if (shared && !last) turn_done(ev, at, rel == 2 * td.nch - 1);
                }
            } else {
                const bool resident = !ganged && td.nch <= L::kResident;
                if (!resident || last) {
                    for (int i = 0; i < td.nch; ++i) {
                        const int rel = ST && i + td.c0 >= td.nch ? i + td.c0 - td.nch : ST ? i + td.c0 : i;
                        const int ev = ST && p.rotate ? td.q0 + rel : rel;
                        const int r = D == 64 ? 0 : resident ? rel : (int)(n++ & 1);
                        if (shared) {
                            if (p.rotate) {
                                at = place(rel);
                                first = at == 0;
                                last = at == td.nch - 1;
                            }
                            ok = turn(ev, at);
                        }
                        ok = ok && mbar_wait_all(bar(kBDq + r), (dq_use >> r) & 1, cta_abort);
                        if (!ok) break;
                        dq_use ^= 1u << r;
                        tc_fence_after();
                        uint32_t v[kLd][32];
#pragma unroll
                        for (int q = 0; q < kLd; ++q) tmem_ld32(tl + L::kColDq + L::kStrideDq * r + 32 * q, v[q]);
                        hand_back(kBDqFree + r);
                        const int slot = rel * kTile + row, u = u0 + slot / RW, a = ST ? unit_row(u, td.ns) : u, b = slot % RW + (ST ? 32 * (u - a * td.ns) : 0);
                        const bool add = !resident && !first, tok = a < td.eh && b < td.ew;
                        uint4* dst = reinterpret_cast<uint4*>(dq + (sample + (tok ? win_token(g, td.wr, td.wc, a, b) : 0)) * g.ts + td.head * D);
#pragma unroll
                        for (int q = 0; q < kLd; ++q) {
                            float4* s4 = slab + (rel * (D / 4) + q * 8) * 128;
                            if (!last || split) {
                                to_slab(s4, v[q], add);
                            } else {
                                if (add) from_slab(s4, v[q]);
                                if (kExchange) store_rows32(dq + 32 * q, tok ? (long long)(dst - reinterpret_cast<uint4*>(dq)) * 8 : -1, v[q], out_scale, lane);
                                else if (tok) store_scaled32(dst + 4 * q, v[q], out_scale);
                            }
                        }
                        if (shared && !last) turn_done(ev, at, rel == td.nch - 1);
                    }
                }
            }
            if (!ok) break;
            if (shared) {
                signal_pending();
                if (!p.rotate && last) signal(flag(p.events), td.use + 1);
            }
            // ---- dV and dK of the key tile
            ok = mbar_wait_all(bar(kBAcc), na & 1, cta_abort);
            if (!ok) break;
            ++na;
            tc_fence_after();
            const int slot = td.kt * kTile + row, u = slot / RW, a = ST ? unit_row(u, td.ns) : u, b = slot % RW + (ST ? 32 * (u - a * td.ns) : 0);
            const bool tok = a < td.eh && b < td.ew;
            const size_t off = (sample + (tok ? win_token(g, td.wr, td.wc, a, b) : 0)) * g.ts + td.head * D;
#pragma unroll
            for (int q = 0; q < D / 32; ++q) {
                uint32_t v[2][32];
                tmem_ld32(tl + L::kColAcc + 64 * q, v[0]);
                tmem_ld32(tl + L::kColAcc + 64 * q + 32, v[1]);
                if (q == D / 32 - 1) hand_back(kBAccFree);
                else tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int c = 2 * q + i;
                    const bool is_k = c >= D / 32;
                    __nv_bfloat16* to = (is_k ? dk : dv) + 32 * (is_k ? c - D / 32 : c);
                    const float f = is_k ? out_scale : 1.f;
                    if (kExchange) store_rows32(to, tok ? (long long)off : -1, v[i], f, lane);
                    else if (tok) store_scaled32(reinterpret_cast<uint4*>(to + off), v[i], f);
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kRegsOther));
        if (warp == kPlanWarp) {
            // -------------------------------------------------------------- tiles in the order every role meets them
            struct { int b, wr, wc; } cur = {0, 0, 0};
            unsigned i = 0;
            bool ok = true;
            auto put = [&](int flags, int head, int eh, int ew, int kt, int nch, int q0, int slab, int seq = 0, int use = 0, int c0 = 0) {
                ok = mbar_wait_all(bar(kBDescFree + i % kDescs), ((i / kDescs) & 1) ^ 1u, cta_abort);
                if (!ok) return;
                if (lane == 0) {
                    int4* dst = reinterpret_cast<int4*>(smem + L::kOffDesc + (i % kDescs) * 64);
                    dst[0] = make_int4(head, cur.b, cur.wr, cur.wc);
                    dst[1] = make_int4(eh, ew, kt, L::kTwo ? nch | q0 << 16 : nch);
                    dst[2] = make_int4((!g.ph && g.sh > 0) ? g.H - g.sh - cur.wr * g.w : (1 << 20), (!g.pw && g.sw > 0) ? g.W - g.sw - cur.wc * g.w : (1 << 20), flags, slab);
                    if (ST) dst[3] = make_int4(strips_of(ew), seq, use, c0);
                    mbar_arrive(bar(kBDesc + i % kDescs));
                }
                __syncwarp();
                ++i;
            };
            // The tables of the tile in front of the last one put: each of its copies takes this warp a few hundred cycles, and
            // the loading warp has as many of its own (with both on one warp it was what the score warp waited for).
            unsigned n = 0;                          // half chunks so far
            int t_head = 0, t_kt = 0, t_nch = 0, t_q0 = 0, t_win = 0;
            auto tables = [&]() {
                // bias rows of half chunk hc: row differences from hc kG - (kt + 1) (128 / RW) + 1 on
                const size_t rows0 = ((size_t)t_head * 2 * p.rmax + p.rmax + 1 - (t_kt + 1) * (kTile / RW)) * (2 * RW);
                const float4* stat = p.rowstat + ((size_t)t_win * g.heads + t_head) * (p.npad / 2);
                for (int hc = 2 * t_q0; ok && hc < 2 * (t_q0 + t_nch); ++hc, ++n) {
                    const int r = (int)(n % L::kTabs);
                    ok = mbar_wait_all(bar(kBTabFree + r), ((n / L::kTabs) & 1) ^ 1u, cta_abort);
                    if (!ok) break;
                    const uint32_t dst = smem0 + L::kOffTab + r * L::kTabB;
                    if (elect_one()) {
                        mbar_arrive_expect_tx(bar(kBTab + r), 512 + 2 * L::kCopyB);
                        bulk_load(dst, stat + hc * 32, 512, bar(kBTab + r));
                        bulk_load(dst + L::kOffCopy0, p.bias0 + rows0 + hc * kG * (2 * RW), L::kCopyB, bar(kBTab + r));
                        bulk_load(dst + L::kOffCopy1, p.bias1 + rows0 + hc * kG * (2 * RW), L::kCopyB, bar(kBTab + r));
                    }
                    __syncwarp();
                }
            };
            const int member = L::kGang ? (int)blockIdx.x % p.gang : 0;
            int seq = 0, windows = 0;                // tiles and windows of several tiles of the gang so far
            for (long long u = L::kGang ? blockIdx.x / p.gang : blockIdx.x; ok && u < p.units; u += L::kGang ? p.gangs : gridDim.x) {
                // unit -> head and share, window, sample (the windows of the launch: see Params)
                const unsigned hs = (unsigned)g.heads << p.split_log2, bottom = (unsigned)(g.Mh - p.row1) * g.Mw;
                const unsigned per_row = p.inner ? p.col1 : g.Mw - p.col1, per_sample = p.row1 * per_row + (p.inner ? 0u : bottom);
                const unsigned wi = (unsigned)u / hs, hd = (unsigned)u - wi * hs;
                cur.b = wi / per_sample;
                unsigned r = wi - cur.b * per_sample;
                if (!p.inner && r < bottom) {
                    cur.wr = p.row1 + r / g.Mw;
                    cur.wc = r % g.Mw;
                } else {
                    if (!p.inner) r -= bottom;
                    cur.wr = r / per_row;
                    cur.wc = (p.inner ? 0 : p.col1) + r % per_row;
                }
                const int head = hd >> p.split_log2, split = hd - (head << p.split_log2);
                const int eh = min(g.w, g.H - cur.wr * g.w), ew = min(g.w, g.W - cur.wc * g.w), nch = (eh * (ST ? strips_of(ew) : 1) * RW + kTile - 1) / kTile;
                const int kt0 = (split * nch) >> p.split_log2, kt1 = ((split + 1) * nch) >> p.split_log2;
                // a slab per CTA; where windows are split, per unit in the order of all windows
                const int slab = p.split_log2 ? (int)((((long long)(cur.b * g.Mh + cur.wr) * g.Mw + cur.wc) * hs) + hd) : p.slab0 + (int)blockIdx.x;
                // where the window is two, a part's tiles meet its own queries only
                const int t0 = !L::kTwo || cur.wr != p.part_row ? 0 : ST ? part_tiles(p.part_ha, eh, strips_of(ew) * RW) : p.part_ha * RW / kTile;
                if (L::kGang && p.gang > 1) {
                    for (int q0 = 0; q0 < nch;) {
                        const int tn = q0 == 0 && t0 > 0 ? t0 : nch - q0;
                        for (int kt = gang_first_tile(member, seq, p.gang); ok && kt < tn; kt += p.gang)
                            put(1 | (kt == 0 ? 2 : 0) | (kt == tn - 1 ? 4 : 0), head, eh, ew, q0 + kt, tn, q0, (int)(blockIdx.x / p.gang) * p.ring + windows % p.ring, seq,
                                windows / p.ring, gang_first_chunk(kt, tn, p.gang, p.rotate));
                        seq += tn;
                        windows += tn > 1;
                        q0 += tn;
                    }
                    continue;
                }
                for (int kt = kt0; ok && kt < kt1; ++kt) {
                    const int q0 = t0 > 0 && kt >= t0 ? t0 : 0, q1 = t0 > 0 && kt < t0 ? t0 : nch;
                    put(1 | (kt == max(kt0, q0) ? 2 : 0) | (kt == min(kt1, q1) - 1 ? 4 : 0), head, eh, ew, kt, q1 - q0, q0, slab);
                    if (L::kTables) {
                        tables();
                        t_head = head; t_kt = kt; t_nch = q1 - q0; t_q0 = q0; t_win = (cur.b * g.Mh + cur.wr) * g.Mw + cur.wc;
                    }
                }
            }
            if (ok) put(0, 0, 0, 0, 0, 0, 0, 0);
            if (L::kTables) tables();
        } else if (warp == kLoaderWarp) {
            // -------------------------------------------------------------- copies.  One warp fills every slot: a wait names a
            // barrier's phase by parity, so a slot's next use may only be waited for by who has filled its last one
            SlotQueue<L::kSlots> sq;
            sq.init();
            uint32_t use = 0;                        // bit per slot: parity of the slot's fills
            bool ok = true;
            // lane -> channel part, window row of a tile or of the two half chunks
            const int part = lane % kParts, row = lane / kParts;
            // one slot; `two`: Q and dO of a half chunk (else the two 64-slot groups of a K or V tile); a0 = first window row
            auto fill = [&](int s, const Maps<ST>& m0, const Maps<ST>& m1, const __nv_bfloat16* x0, const __nv_bfloat16* x1, int a0, bool two) {
                ok = mbar_wait_all(bar(kBEmpty + s), ((use >> s) & 1) ^ 1u, cta_abort);
                if (!ok) return;
                use ^= 1u << s;
                const bool fix = D == 32 && p.cols.skip && td.wc == p.cols.seam;
                // ST: whether the seam cuts strip u
                auto cut = [&](int u) { return !ST || u - unit_row(u, td.ns) * td.ns == p.cols.n1 >> 5; };
                if (D == 32 && fix) {
                    // the seam column's slot n1 cannot be the start of a bulk copy of 64-byte rows (128-byte alignment)
                    for (int i = lane; i < 2 * kG * 4; i += 32) {
                        const int h = i / (kG * 4), r = (i / 4) % kG, ch = i & 3, u = a0 + (two ? r : h * kG + r), a = ST ? unit_row(u, td.ns) : u;
                        if (!cut(u)) continue;
                        const int tstride = (two && h) ? g.heads * D : g.ts;
                        uint4 val = make_uint4(0, 0, 0, 0);
                        if (a < td.eh && p.cols.n1 < td.ew)
                            val = __ldg(reinterpret_cast<const uint4*>((h ? x1 : x0) + ((size_t)td.b * g.H * g.W + win_token(g, td.wr, td.wc, a, p.cols.n1)) * tstride + td.head * D) + ch);
                        // rows of a K / V tile: both groups in one region; Q and dO: a region each
                        const int rr = (two ? r : h * kG + r) * RW + (ST ? p.cols.n1 & 31 : p.cols.n1);
                        *reinterpret_cast<uint4*>(smem + s * L::kSlotB + (two ? h * kHalf * D * 2 : 0) + tile_off<32>(rr, ch)) = val;
                    }
                    fence_proxy_async();
                    __syncwarp();
                }
                const uint32_t base = smem0 + s * L::kSlotB;
                if constexpr (ST) {
                    // 64 slots of a window row are one copy where the strips are even in number, a strip one where they are not
                    const bool whole = (td.ns & 1) == 0 && td.wc != p.cols.seam && td.wc < p.cols.first_wrapped && td.wc != p.cols.last;
                    if (lane == 0) {
                        int n = 0;
                        if (fix) n = two ? 2 * (cut(a0) + cut(a0 + 1)) : cut(a0) + cut(a0 + 1) + cut(a0 + 2) + cut(a0 + 3);
                        mbar_arrive_expect_tx(bar(kBFull + s), L::kSlotB - n * kRowB);
                    }
                    __syncwarp();
                    if (row < (whole ? 2 : 4)) {
                        const int second = whole ? row : row >> 1, r = whole ? 0 : row & 1;           // of two: the tensor, else the 64-slot group
                        const int u = a0 + r + (two ? 0 : 2 * second), a = unit_row(u, td.ns), st = u - a * td.ns;
                        const uint32_t dst = base + r * 32 * kRowB + (two ? second * kHalf * D * 2 + part * kHalf * kRowB : part * kTile * kRowB + second * kHalf * kRowB);
                        const Maps<ST>& m = second ? m1 : m0;
                        if (whole) {
                            int y = td.wr * g.w + a + g.sh;
                            if (y >= g.H) y -= g.H;
                            tma_load_4d(dst, &m.group, td.head * D + part * L::kPartCh, 32 * st, td.wc, a < td.eh ? td.b * g.H + y : g.B * g.H, bar(kBFull + s));
                        } else {
                            load_win_strip<kRowB>(m, p.cols, dst, g, td.b, td.wr, td.wc, td.eh, a, st, td.head * D + part * L::kPartCh, bar(kBFull + s));
                        }
                    }
                } else if (win_group_whole<RW>(p.cols, g, td.wr, td.wc, td.eh, a0, two ? 1 : 2)) {
                    // the common case: one thread, one copy per group and channel part
                    if (elect_one()) {
                        mbar_arrive_expect_tx(bar(kBFull + s), L::kSlotB);
                        int y0 = td.wr * g.w + a0 + g.sh;
                        if (y0 >= g.H) y0 -= g.H;
                        y0 += td.b * g.H;
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int pt = 0; pt < kParts; ++pt)
                                tma_load_4d(base + (two ? h * kHalf * D * 2 + pt * kHalf * kRowB : pt * kTile * kRowB + h * kHalf * kRowB), &(h ? m1 : m0).group,
                                            td.head * D + pt * L::kPartCh, 0, td.wc, y0 + (two ? 0 : h * kG), bar(kBFull + s));
                    }
                } else {
                    if (lane == 0) mbar_arrive_expect_tx(bar(kBFull + s), L::kSlotB - (fix ? 2 * kG * kRowB : 0));
                    __syncwarp();
                    if (row < 2 * kG) {
                        const int second = row / kG, r = row % kG;
                        const uint32_t dst = base + r * RW * kRowB + (two ? second * kHalf * D * 2 + part * kHalf * kRowB : part * kTile * kRowB + second * kHalf * kRowB);
                        load_win_row<RW, kRowB>(second ? m1 : m0, p.cols, dst, g, td.b, td.wr, td.wc, td.eh, a0 + (two ? r : row),
                                                td.head * D + part * L::kPartCh, bar(kBFull + s));
                    }
                }
                __syncwarp();
            };
            while (ok && next_tile()) {
                const int sk = sq.pop(), sv = sq.pop();
                fill(sk, mk, mk, p.k, p.k, td.kt * 2 * kG, false);
                if (ok) fill(sv, mv, mv, p.v, p.v, td.kt * 2 * kG, false);
                for (int i = 0; ok && i < 2 * td.nch; ++i) {
                    const int hc = 2 * td.q0 + (ST && i + 2 * td.c0 >= 2 * td.nch ? i + 2 * td.c0 - 2 * td.nch : ST ? i + 2 * td.c0 : i);
                    fill(sq.take_half(), mq, mg, p.q, p.d_o, hc * kG, true);
                }
                sq.end_tile(sk, sv);
            }
        } else if (warp == kScoreWarp) {
            // -------------------------------------------------------------- S^T and dP^T
            constexpr uint32_t kIdS = make_idesc_elem(128, kHalf, 0, 0);
            const uint64_t d_k = D == 32 ? make_sdesc_sw64(smem0, 512) : make_sdesc_sw128(smem0);       // K-major rows
            const uint32_t hi = sdesc_hi(d_k), lo = sdesc_lo(d_k);
            constexpr int kPerPart = L::kPartCh / 16;
            SlotQueue<L::kSlots> sq;
            sq.init();
            uint32_t full_use = 0;
            unsigned n = 0;                          // pairs of half chunks so far
            bool ok = true;
            auto wait_full = [&](int s) {
                ok = ok && mbar_wait_all(bar(kBFull + s), (full_use >> s) & 1, cta_abort);
                full_use ^= 1u << s;
            };
            while (ok && next_tile()) {
                const int sk = sq.pop(), sv = sq.pop();
                wait_full(sk);
                wait_full(sv);
                const uint32_t ak = lo + sk * (L::kSlotB >> 4), av = lo + sv * (L::kSlotB >> 4);
                for (int hc = 0; ok && hc < 2 * td.nch; hc += 2, ++n) {
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        const int s = sq.take_half();
                        wait_full(s);
                        // the buffer's last scores have been read (head dim 128: P^T by its product)
                        ok = ok && mbar_wait_all(bar((L::kOwnP ? kBSFree : kBPFree) + b), (n & 1) ^ 1u, cta_abort);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t bq = lo + s * (L::kSlotB >> 4), bg = bq + kHalf * D * 2 / 16;
                        const uint32_t ds = tmem + 128u * b;
                        auto scores = [&](uint32_t d, uint32_t a, uint32_t bb) {
#pragma unroll
                            for (int ks = 0; ks < D / 16; ++ks) {
                                const uint32_t oa = (ks / kPerPart) * (kTile * kRowB / 16) + (ks % kPerPart) * 2, ob = (ks / kPerPart) * (kHalf * kRowB / 16) + (ks % kPerPart) * 2;
                                if (ks == 0) mma_ss_h<false>(d, a + oa, bb + ob, hi, kIdS);
                                else mma_ss_h<true>(d, a + oa, bb + ob, hi, kIdS);
                            }
                        };
                        if (elect_one()) {
                            scores(ds, ak, bq);
                            if (D != 128) scores(ds + 64, av, bg);
                        }
                        __syncwarp();
                        // head dim 128: dQ^T of the buffer's last half chunk lies over dP^T.  Head dims 32 and 64: the elementwise
                        // warps may write P^T and dS^T once the last products (head dim 64, buffer 1: and the read-out of dQ,
                        // which lies over them) are done; waiting here, behind the issue, spares them that wait
                        ok = mbar_wait_all(bar(D == 128 || (D == 64 && b == 1) ? (D == 128 ? kBDqFree + b : kBDqFree) : kBPFree + b), (n & 1) ^ 1u, cta_abort);
                        if (!ok) break;
                        tc_fence_after();
                        if (elect_one()) {
                            if (D == 128) scores(ds + 64, av, bg);
                            mma_commit(bar(kBSdp + b));
                        }
                        __syncwarp();
                    }
                }
                sq.end_tile(sk, sv);
            }
        } else if (warp == kProductWarp) {
            // -------------------------------------------------------------- dV, dK, dQ
            constexpr uint32_t kIdAcc = make_idesc_elem(128, D, 0, 1);
            constexpr uint32_t kIdQ = D == 128 ? make_idesc_elem(128, kHalf, 1, 1) : make_idesc_elem(128, D, 1, 1);
            const uint64_t d_half = D == 32 ? make_sdesc_sw64_mn(smem0, 512, 512) : make_sdesc_sw128(smem0, kHalf * kRowB);   // Q, dO rows as B
            const uint64_t d_tile = D == 32 ? make_sdesc_sw64_mn(smem0, 512, 512) : make_sdesc_sw128(smem0, kTile * kRowB);   // K rows as B (or A)
            const uint64_t d_ds = make_sdesc_sw128(smem0 + L::kOffDs, L::kDsB);                                               // dS^T tiles, 64 queries each
            const uint32_t hi = sdesc_hi(d_half), hi_ds = sdesc_hi(d_ds), lo_half = sdesc_lo(d_half), lo_tile = sdesc_lo(d_tile), lo_ds = sdesc_lo(d_ds);
            constexpr uint32_t kStep = 16 * kRowB / 16;          // 16 rows, in units of 16 bytes
            SlotQueue<L::kSlots> sq;
            sq.init();
            unsigned n = 0, na = 0, ev = 0;          // pairs of half chunks, key tiles, dQ events outside windows that keep it
            uint32_t dq_free = 0;
            bool ok = true;
            while (ok && next_tile()) {
                const int sk = sq.pop(), sv = sq.pop();
                const bool resident = !(L::kGang && p.gang > 1) && td.nch <= L::kResident, fresh = !resident || (td.flags & 2), ready = !resident || (td.flags & 4);
                const uint32_t acc = tmem + L::kColAcc, kt_lo = lo_tile + sk * (L::kSlotB >> 4);
                for (int hc = 0; ok && hc < 2 * td.nch; hc += 2, ++n) {
#pragma unroll
                    for (int b = 0; b < 2; ++b) {
                        const int s = sq.take_half();
                        const bool first = b == 0 && hc == 0, last = b == 1 && hc + 2 == 2 * td.nch;
                        ok = mbar_wait_all(bar(kBDs + b), n & 1, cta_abort);
                        if (ok && first) ok = mbar_wait_all(bar(kBAccFree), (na & 1) ^ 1u, cta_abort);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t bq = lo_half + s * (L::kSlotB >> 4), bg = bq + kHalf * D * 2 / 16;
                        const uint32_t ap = tmem + L::kColP + L::kStrideP * b, ads_t = ap + L::kDsOff;
                        if (elect_one()) {
                            if (first) mma_ts_h<false>(acc, ap, bg, hi, kIdAcc);
                            else mma_ts_h<true>(acc, ap, bg, hi, kIdAcc);
#pragma unroll
                            for (int ks = 1; ks < 4; ++ks) mma_ts_h<true>(acc, ap + (ks >> 1) * L::kPieceP + (ks & 1) * 8, bg + ks * kStep, hi, kIdAcc);
                            if (D == 128) mma_commit(bar(kBPFree + b));           // S^T of the next half chunk may follow
                            if (first) mma_ts_h<false>(acc + D, ads_t, bq, hi, kIdAcc);
                            else mma_ts_h<true>(acc + D, ads_t, bq, hi, kIdAcc);
#pragma unroll
                            for (int ks = 1; ks < 4; ++ks) mma_ts_h<true>(acc + D, ads_t + (ks >> 1) * L::kPieceP + (ks & 1) * 8, bq + ks * kStep, hi, kIdAcc);
                            if (D != 128) mma_commit(bar(kBPFree + b));
                            if (D == 128) {
                                const uint32_t dst = tmem + 128u * b + L::kColDq, bds = lo_ds + b * (L::kDsB >> 4);
                                mma_ss_h<false>(dst, kt_lo, bds, hi, kIdQ);
#pragma unroll
                                for (int ks = 1; ks < 8; ++ks) mma_ss_h<true>(dst, kt_lo + ks * 128, bds + ks * 128, hi, kIdQ);
                                mma_commit(bar(kBDq + b));
                            }
                            if (!last) mma_commit(bar(kBEmpty + s));
                        }
                        __syncwarp();
                        if (D != 128 && b == 1) {
                            const int r = D == 64 ? 0 : resident ? hc >> 1 : (int)(ev++ & 1);
                            if (D == 32 && fresh) {
                                ok = mbar_wait_all(bar(kBDqFree + r), ((dq_free >> r) & 1) ^ 1u, cta_abort);
                                dq_free ^= 1u << r;
                                if (!ok) break;
                                tc_fence_after();
                            }
                            const uint32_t dcol = tmem + L::kColDq + L::kStrideDq * r, ads = lo_ds + (n & 1) * (2 * L::kDsB >> 4);
                            if (elect_one()) {
                                if (fresh) mma_ss_hh<false>(dcol, ads, hi_ds, kt_lo, hi, kIdQ);
                                else mma_ss_hh<true>(dcol, ads, hi_ds, kt_lo, hi, kIdQ);
#pragma unroll
                                for (int ks = 1; ks < 8; ++ks) mma_ss_hh<true>(dcol, ads + ks * 128, hi_ds, kt_lo + ks * kStep, hi, kIdQ);
                                if (ready) mma_commit(bar(kBDq + r));
                            }
                            __syncwarp();
                        }
                        if (last && elect_one()) {
                            mma_commit(bar(kBAcc));
                            mma_commit(bar(kBEmpty + s));
                            mma_commit(bar(kBEmpty + sv));
                            mma_commit(bar(kBEmpty + sk));
                        }
                        __syncwarp();
                    }
                }
                sq.end_tile(sk, sv);
                ++na;
            }
        }
    }

    // teardown: every role ends up here, also after an expired wait
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kProductWarp) tmem_dealloc(tmem, 512);
    if (KIND == 1 && p.overlap) wait_for_prerequisites();
    if (tid == 0 && *cta_abort) atomicExch(&g_bwd_onepass_timeout, 1);
}

// Everything the kernel above reads besides q, k, v and dO, in one launch.  Blocks [0, stat_blocks): per slot of a window
// -lse log2 e and delta = rowsum(dO O), by windows and slots (slots without a token: -inf and 0), 64 slots x up to 16 heads
// a block: as many as leave four blocks an SM.  Bound by the reads of O and dO, on small grids by the chain of a
// block's reads (42 x 42 tokens, 13 x 128, side 21: 16 heads a block 29 us; so 10).  The other blocks: the bias tables by row difference and diagonal, and the
// zeroed bias-gradient table.
constexpr int kStatHeads = 16;

template <int D, int RW, bool ST, bool FEW>
__global__ void __launch_bounds__(256)
swin_bwd_onepass_prep_kernel(const Geo g, const __nv_bfloat16* __restrict__ o, const __nv_bfloat16* __restrict__ d_o, const float* __restrict__ lse,
                             const float* __restrict__ bias, float4* __restrict__ rowstat, float* __restrict__ bias0, float* __restrict__ bias1,
                             float* __restrict__ dbias_acc, int npad, int rmax, int rl, unsigned stat_blocks, int few_heads, unsigned* __restrict__ flags, int n_flags) {
    if (blockIdx.x >= stat_blocks) {
        for (int i = (blockIdx.x - stat_blocks) * 256 + threadIdx.x; i < n_flags; i += (gridDim.x - stat_blocks) * 256) flags[i] = 0;
        const int per_head = 2 * rmax * rl, total = per_head * g.heads, nw = 2 * g.w - 1;
        for (int i = (blockIdx.x - stat_blocks) * 256 + threadIdx.x; i < total; i += (gridDim.x - stat_blocks) * 256) {
            // (the larger tables: neighbouring threads read neighbouring heads)
            const int head = ST ? i % g.heads : i / per_head, e = ST ? i / g.heads : i - head * per_head, at = head * per_head + e;
            const int da = e / rl - rmax, db = e % rl - rl / 2;
            const bool row = da > -g.w && da < g.w;
            const float* src = bias + ((size_t)(da + g.w - 1) * nw + db + g.w - 1) * g.heads + head;
            bias0[at] = row && db > -g.w && db < g.w ? kLog2e * __ldg(src) : 0.f;
            bias1[at] = row && db + 1 > -g.w && db + 1 < g.w ? kLog2e * __ldg(src + g.heads) : 0.f;
            dbias_acc[at] = 0.f;
        }
        return;
    }
    constexpr int kLanes = D / 8, kRowsPass = 256 / kLanes;
    __shared__ float4 st[kStatHeads][33];
    const int block_heads = FEW ? few_heads : kStatHeads;
    const unsigned hgroups = (g.heads + block_heads - 1) / block_heads, chunks = npad / 64;
    unsigned x = blockIdx.x;
    const int h0 = (int)(x % hgroups) * block_heads;
    x /= hgroups;
    const int chunk = (int)(x % chunks);
    x /= chunks;
    const int wc = (int)(x % g.Mw), wr = (int)(x / g.Mw % g.Mh), b = (int)(x / g.Mw / g.Mh);
    const int nh = min(block_heads, g.heads - h0), eh = min(g.w, g.H - wr * g.w), ew = min(g.w, g.W - wc * g.w);
    const int l = threadIdx.x % kLanes;
    for (int r0 = 0; r0 < 64 * nh; r0 += kRowsPass) {
        const int r = r0 + threadIdx.x / kLanes;
        const int s = r / nh, h = r - s * nh, slot = chunk * 64 + s, u = slot / RW, ns = strips_of(ew), a = ST ? unit_row(u, ns) : u, bb = slot % RW + (ST ? 32 * (u - a * ns) : 0);
        const bool in = r < 64 * nh, tok = in && a < eh && bb < ew;
        float dot = 0.f, nl2 = -INFINITY;
        if (tok) {
            const size_t row = ((size_t)b * g.H * g.W + win_token(g, wr, wc, a, bb)) * g.heads + h0 + h;
            const uint4 x0 = __ldg(reinterpret_cast<const uint4*>(o + row * D) + l), x1 = __ldg(reinterpret_cast<const uint4*>(d_o + row * D) + l);
            const uint32_t xa[4] = {x0.x, x0.y, x0.z, x0.w}, xb[4] = {x1.x, x1.y, x1.z, x1.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float2 fa = elem2_to_float2(xa[i]), fb = elem2_to_float2(xb[i]);
                dot += fa.x * fb.x + fa.y * fb.y;
            }
            if (l == 0) nl2 = -kLog2e * __ldg(lse + row);
        }
#pragma unroll
        for (int m = kLanes / 2; m > 0; m >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, m);
        if (in && l == 0) {
            float* dst = reinterpret_cast<float*>(&st[h][s >> 1]) + (s & 1);
            dst[0] = nl2;
            dst[2] = dot;
        }
    }
    __syncthreads();
    float4* dst = rowstat + (((size_t)b * g.Mh * g.Mw + wr * g.Mw + wc) * g.heads + h0) * (npad / 2) + chunk * 32;
    for (int i = threadIdx.x; i < nh * 32; i += 256) dst[(size_t)(i >> 5) * (npad / 2) + (i & 31)] = st[i >> 5][i & 31];
}

// dbias[(da, db), head] from the heads' tables; where windows were split, dQ as the sum of their units' slabs in a fixed order.
template <int D, int RW>
__global__ void __launch_bounds__(256)
swin_bwd_onepass_finish_kernel(const Geo g, const float* __restrict__ dbias_acc, float* __restrict__ dbias, const float4* __restrict__ slabs,
                               __nv_bfloat16* __restrict__ dq, int npad, int rmax, int rl, int split_log2, unsigned bias_blocks) {
    wait_for_prerequisites();
    if (blockIdx.x < bias_blocks) {
        const int nw = 2 * g.w - 1, i = blockIdx.x * 256 + threadIdx.x;
        if (i >= nw * nw * g.heads) return;
        const int head = i % g.heads, r = i / g.heads, da = r / nw - (g.w - 1), db = r % nw - (g.w - 1);
        dbias[i] = dbias_acc[((size_t)head * 2 * rmax + da + rmax) * rl + db + rl / 2];
        return;
    }
    const int per_item = npad * D / 4, blocks = (per_item + 255) / 256;
    const unsigned x = blockIdx.x - bias_blocks;
    const long long item = x / blocks;
    const int i = (int)(x % blocks) * 256 + threadIdx.x;
    const int head = (int)(item % g.heads);
    const long long win = item / g.heads;
    const int wc = (int)(win % g.Mw), wr = (int)(win / g.Mw % g.Mh), b = (int)(win / g.Mw / g.Mh);
    const int eh = min(g.w, g.H - wr * g.w), ew = min(g.w, g.W - wc * g.w), nch = (eh * RW + kTile - 1) / kTile;
    const int row = i & 127, cg = i >> 7;
    const int slot0 = D == 128 ? 4 * cg : (cg / (D / 4)) * kTile + row;
    if (i >= per_item || slot0 >= nch * kTile) return;
    const int t0 = Lay<D, RW>::kTwo ? part_tiles((!g.ph && g.sh > 0) ? g.H - g.sh - wr * g.w : (1 << 20), eh, RW) : 0;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    auto add = [&](int s) {
        const float4 t = __ldcg(slabs + ((item << split_log2) + s) * per_item + i);
        v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
    };
    if (t0 == 0) {
        for (int s = 0; s < (1 << split_log2); ++s)
            if (((s * nch) >> split_log2) != (((s + 1) * nch) >> split_log2)) add(s);
    } else {
        // two parts: the slabs of those whose tiles meet the chunk
        const int c_lo = slot0 >= t0 * kTile ? t0 : 0, c_hi = slot0 < t0 * kTile ? t0 : nch;
        for (int s = 0; s < (1 << split_log2); ++s)
            if (max((s * nch) >> split_log2, c_lo) < min(((s + 1) * nch) >> split_log2, c_hi)) add(s);
    }
    const float f = g.scale_log2e * kLn2;
    const uint32_t lo = pack_elem(v.x * f, v.y * f), hi = pack_elem(v.z * f, v.w * f);
    const size_t sample = (size_t)b * g.H * g.W;
    if (D == 128) {
        const uint16_t e[4] = {(uint16_t)lo, (uint16_t)(lo >> 16), (uint16_t)hi, (uint16_t)(hi >> 16)};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int a = (slot0 + k) / RW, bb = (slot0 + k) % RW;
            if (a < eh && bb < ew)
                *reinterpret_cast<uint16_t*>(dq + (sample + win_token(g, wr, wc, a, bb)) * g.ts + head * D + row) = e[k];
        }
    } else {
        const int a = slot0 / RW, bb = slot0 % RW;
        if (a < eh && bb < ew)
            *reinterpret_cast<uint2*>(dq + (sample + win_token(g, wr, wc, a, bb)) * g.ts + head * D + 4 * (cg % (D / 4))) = make_uint2(lo, hi);
    }
}

}  // namespace

cudaError_t read_bwd_onepass_status(int* timed_out) {
    int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(timed_out, g_bwd_onepass_timeout, sizeof(int));
    if (e != cudaSuccess) return e;
    if (*timed_out) e = cudaMemcpyToSymbol(g_bwd_onepass_timeout, &zero, sizeof(int));
    return e;
}

#ifndef TERRA_ELEM_F16
// Bias-table rows run from -table_rmax to table_rmax - 1 and are table_rl floats long.
static int table_rmax(const Geo& g) {
    const int kr = kTile / win_row_slots(g);
    return win_strips(g) ? g.w + 4 : (g.w + kr - 1) / kr * kr;      // (strips: the last key tile's rows reach up to 3 past the window's)
}
static int table_rl(const Geo& g) { return win_strips(g) ? 64 * strips_of(g.w) : 2 * win_row_slots(g); }

bool bwd_onepass_supported(const Geo& g) {
    // entries of the bias tables are numbered in 32 bits, with room for a loop that steps past the last (side 128: 31759 heads)
    if ((long long)g.heads * 2 * table_rmax(g) * table_rl(g) > 0x7ff00000LL) return false;
    // (head dim 32 with sides up to 16 has a kernel of its own, 1.83 against 2.5 ms on the 510 x 1080 grid with 12 heads)
    // Register tiles / this kernel, us, on 240 x 360, 2 x 121 x 250 and 96 x 180 tokens: head dim 64, side 9 676/752 659/719 166/166, 10 572/626 560/601
    // 146/140; 11 517/537 480/496 140/126 (level), 12 1032/451; head dim 128, side 9 889/800 1215/1130 289/263; head dim 32, side 17 948/967
    // 1798/1711 389/406 (level), 18 1126/816 2278/1496 468/384.
    // Strips: where the windows' work in them (strip_work) is at most 10, 9 and 7 times the dense one at head dims 32, 64 and 128: all but windows of
    // few columns.  Register tiles / strips, us: 240 x 360, 6 x 32, side 33 7573/2785; 200 x 64 x 1, 6 x 32, side 64 220/8166; 8 x 128 x 4, 12 x 128, side 64
    // 400/2952; 200 x 8 x 8, 4 x 128, side 40 159/374.  On 1662 shapes strips alone were more than 5 % slower on 243, the rule is wrong on 45.
    if (win_strips(g)) {
        const StripWork x = strip_work(g);
        if (x.strips > (g.d == 32 ? 10 : g.d == 64 ? 9 : 7) * x.dense) return false;
        return g.w <= kMaxWinW && (long long)g.B * g.H * g.W < 0x7fffffffLL && (long long)g.B * g.Mh * g.Mw * g.heads * 128 < 0x7fffffffLL;
    }
    return ((g.d == 64 && g.w > 10) || g.d == 128 || (g.d == 32 && g.w > 16)) && g.w > 8 && g.w <= kMaxOnePassW && (long long)g.B * g.H * g.W < 0x7fffffffLL &&
           (long long)g.B * g.Mh * g.Mw * g.heads * 8 < 0x7fffffffLL;
}

// Gangs (see Params).  The CTAs of a gang read the same Q and dO and add to the same slab a few turns after one another, so these pass
// between L2 and memory once for kGangMin CTAs or more.  The time of a run in a full window's key tiles: the longest gang's windows times their tiles over its
// CTAs, plus half of what its last CTA is behind its first, `lag` a CTA (none of it where they rotate).  The longer that is against a tile the more
// its CTAs wait for turns, a quarter of it beyond 0.3 tiles, whether a window has as many tiles or not.  Gangs of 4, 8, 12, 16, 37 and 74, ms: 128 windows of side
// 64 (heads and windows) at head dim 128 4.38, 4.44, 4.62, 4.98, 6.13, 7.59; 320 10.9, 11.0, 11.4, 12.1, 15.5, 18.6; 64 of side 128 33.9, 34.2, 33.5, 34.0, 33.7, 37.7.
// Over 56 sizes of complete windows what is chosen is at most 10 % from the best.
static void plan_gangs(OnePassPlan& p, const Geo& g, long long items, int tiles) {
    p.gangs = kPlanSms;
    p.gang = p.ring = 1;
    p.rotate = p.flags = 0;
    if (!p.strips) return;
    // Up to six windows a gang: what each takes (its parts' tiles, against their own queries) in the order in which the gangs take them; of more
    // all count as full.
    constexpr int kMostGangs = kPlanSms / kGangMin, kListed = 6 * kMostGangs;
    double share[kListed];
    int parts[kListed][2];
    if (items <= kListed) {
        const int ha = !g.ph && g.sh > 0 ? (g.H - g.sh) % g.w : 0, part_row = ha > 0 ? (g.H - g.sh) / g.w : -1;
        for (int i = 0; i < items; ++i) {
            const int win = i / g.heads % (g.Mh * g.Mw), wr = win / g.Mw, wc = win % g.Mw, eh = wr < g.H / g.w ? g.w : g.H % g.w;
            const int slots = strips_of(wc < g.W / g.w ? g.w : g.W % g.w) * p.rw, all = (eh * slots + kTile - 1) / kTile;
            parts[i][0] = wr == part_row ? part_tiles(ha, eh, slots) : 0;
            parts[i][1] = all - parts[i][0];
            share[i] = ((double)parts[i][0] * parts[i][0] + (double)parts[i][1] * parts[i][1]) / tiles;
        }
    }
    // Where every gang has one window its CTAs go by whole tiles, have no chain from one window to the next (119 x 303 tokens, 3 x 128, side 64: 30 gangs
    // of 4 1105 us, 15 of 9 1322; 63 x 123, 12 x 128, side 128: 12 of 12 1636, 6 of 24 2020) and read Q, dO and slab (`held`: of the parts worked on) all
    // over, each for itself where L2 does not hold them (128 x 128, 16 x 64, side 128, 134 MB: 16 gangs of 9 1.22 times as long as 8 of 18; 16 x 32, 67 MB: 1.02).
    double held = 0;
    for (int i = 0; items <= kListed && i < items; ++i) held += 8.0 * kTile * g.d * (parts[i][0] > parts[i][1] ? parts[i][0] : parts[i][1]);
    const double lag = kGangLag / (2.0 * tiles);
    double best = 0;
    for (int n = 1; n <= items && n <= kMostGangs; ++n) {
        const int s = kPlanSms / n;
        const double behind = lag * s, slow = behind > 0.3 ? 1 + 0.25 * (behind - 0.3) : 1;
        double longest = items <= kListed ? 0 : (double)((items + n - 1) / n) * tiles / s;
        for (int k = 0; items <= kListed && k < n && (n == 1 || n == items || slow * longest <= best); ++k) {      // (no further than until it is longer)
            double x = 0;
            if (n == items)
                for (int t : parts[k]) x += (double)((t + s - 1) / s) * t / tiles;
            else
                for (int i = k; i < items; i += n) x += share[i];
            if (n < items) x /= s;
            if (x > longest) longest = x;
        }
        const double t = n == items ? (held < (s > 4 ? 115e6 : 160e6) ? 0.9 : 1.2) * longest : slow * longest + 0.5 * behind;
        if (n == 1 || t <= best) { best = t; p.gangs = n; p.gang = s; }
    }
    const long long most = (items + p.gangs - 1) / p.gangs * tiles;
    if (p.gang > most) p.gang = (int)most;
    p.rotate = items <= p.gangs;
    if (p.rotate) p.gang = (tiles + (tiles + p.gang - 1) / p.gang - 1) / ((tiles + p.gang - 1) / p.gang);      // as many tiles for each
    // from a window's first tile to its last one's end, over the time between two windows
    const int turn = p.gang < tiles ? p.gang : tiles;
    p.ring = p.rotate ? 1 : (int)std::ceil(((tiles + p.gang - 1) / p.gang + lag * turn) * p.gang / tiles) + 1;
    p.flags = p.gang > 1 ? p.gangs * p.ring * ((p.npad / (g.d == 128 ? 64 : 128)) + 1) * 4 : 0;      // (more than the turns need; a gang of one takes none)
}

// The plan's gangs on `ctas` CTAs at a time: smaller gangs, then fewer; with several windows a gang its CTAs go after one another.  On one CTA the
// windows have it in turn, with a slab of the first gang's.
GangShape fit_gangs(const OnePassPlan& p, long long units, int ctas) {
    GangShape s = {p.gangs, p.gang, p.rotate};
    if (s.gangs * s.gang > ctas) {
        s.gang = ctas / s.gangs > 2 ? ctas / s.gangs : ctas < 2 ? 1 : 2;
        s.gangs = s.gangs < ctas / s.gang ? s.gangs : ctas / s.gang;
    }
    if (s.gangs < units || s.gang == 1) s.rotate = 0;
    return s;
}

// SMs that a launch in `stream` may use: a green context's stream has a part of the device.
int sms_of_stream(cudaStream_t stream, int device_sms) {
    using GreenOfStream = CUresult (*)(CUstream, CUgreenCtx*);
    using ResourceOfGreen = CUresult (*)(CUgreenCtx, CUdevResource*, CUdevResourceType);
    struct Entries { GreenOfStream green; ResourceOfGreen resource; };
    static const Entries e = [] {
        Entries x = {nullptr, nullptr};
        void *a = nullptr, *b = nullptr;
        cudaDriverEntryPointQueryResult qa, qb;
        if (cudaGetDriverEntryPoint("cuStreamGetGreenCtx", &a, cudaEnableDefault, &qa) == cudaSuccess && qa == cudaDriverEntryPointSuccess &&
            cudaGetDriverEntryPoint("cuGreenCtxGetDevResource", &b, cudaEnableDefault, &qb) == cudaSuccess && qb == cudaDriverEntryPointSuccess)
            x = {reinterpret_cast<GreenOfStream>(a), reinterpret_cast<ResourceOfGreen>(b)};
        return x;
    }();
    CUgreenCtx ctx = nullptr;
    CUdevResource r;
    if (!e.green || e.green(stream, &ctx) != CUDA_SUCCESS || !ctx || e.resource(ctx, &r, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS) return device_sms;
    const int sms = (int)r.sm.smCount;
    return sms < 1 || sms > device_sms ? device_sms : sms;
}

OnePassPlan bwd_onepass_plan(const Geo& g) {
    OnePassPlan p;
    p.rw = win_row_slots(g);
    const int rows = g.w < g.H ? g.w : g.H;
    p.strips = win_strips(g) ? strips_of(g.w) : 0;
    const int tiles = (rows * (p.strips ? strips_of(g.w < g.W ? g.w : g.W) : 1) * p.rw + kTile - 1) / kTile;
    p.npad = tiles * kTile;
    p.rl = table_rl(g);
    p.rmax = table_rmax(g);
    // Units per window: as many as keep the SMs busy.  The time of a launch is the number of unit rounds x key tiles per
    // unit; splitting costs a sum over slabs, so it has to save an eighth of that time.
    const long long items = (long long)g.B * g.Mh * g.Mw * g.heads;
    p.split_log2 = 0;
    double best = 0;
    for (int ls = 0; ls <= (p.strips ? 0 : 3) && (1 << ls) <= tiles; ++ls) {
        const double t = (double)(((items << ls) + kPlanSms - 1) / kPlanSms) * ((tiles + (1 << ls) - 1) >> ls);
        if (ls == 0 || t < 0.875 * best) { best = t; p.split_log2 = ls; }
    }
    p.units = items << p.split_log2;
    plan_gangs(p, g, items, tiles);
    const int most = (g.d == 128 ? 1 : 2) * kMaxCtas;    // CTAs of the launches that may overlap (see launch_onepass)
    const size_t ctas = p.units < most ? (size_t)p.units : (size_t)most;
    const size_t slabs = p.split_log2 ? (size_t)p.units : p.strips && p.gang > 1 ? (size_t)p.gangs * p.ring : ctas;
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    const size_t table = up(sizeof(float) * (size_t)g.heads * 2 * p.rmax * p.rl);
    p.off_bias0 = up(sizeof(float4) * (size_t)g.B * g.Mh * g.Mw * g.heads * (p.npad / 2));
    p.off_bias1 = p.off_bias0 + table;
    p.off_acc = p.off_bias1 + table;
    p.off_slabs = p.off_acc + table;
    // a window whose dQ is complete after one key tile, or stays in TMEM (head dim 32 without strips: Lay::kResident), needs no slab
    const bool slab = p.split_log2 > 0 || g.d != 32 || p.strips ? tiles > 1 : tiles > 2;
    p.bytes = p.off_slabs + (slab ? up(sizeof(float) * slabs * p.npad * g.d) : 0);
    p.off_flags = p.bytes;
    p.bytes += up(sizeof(unsigned) * p.flags);
    return p;
}

bool make_win_cols(WinCols* c, const Geo& g) {
    const int P = g.W - g.sw;                           // where the seam lies in the shifted frame
    c->seam = -1; c->n1 = 0; c->first_wrapped = g.Mw; c->last = -1; c->skip = 0;
    if (g.sw > 0) {
        const int wcs = P / g.w;
        c->n1 = P - wcs * g.w;
        c->first_wrapped = wcs + (c->n1 > 0);
        if (c->n1 > 0) c->seam = wcs;
        c->skip = g.d == 32 && (c->n1 & 1);
    }
    if (g.W % g.w && c->seam != g.Mw - 1) c->last = g.Mw - 1;
    return true;
}

bool make_win_maps(WinMaps* m, const WinCols& c, const Geo& g, const void* base, int ts) {
    std::memset(m, 0, sizeof *m);
    const int rw = win_row_slots(g), box_ch = g.d >= 64 ? 64 : 32;
    const bool st = win_strips(g);
    auto enc = [&](CUtensorMap* out, int col0, int nb, int ncols, int box_b, int box_rows) {
        const char* b = reinterpret_cast<const char*>(base) + (size_t)col0 * ts * 2;
        return encode_win_map(out, g, b, ts, nb, ncols, box_ch, box_b, box_rows);
    };
    int n_main = c.seam >= 0 ? c.seam : c.first_wrapped;
    if (c.last >= 0 && c.last < n_main) n_main = c.last;
    bool ok = true;
    if (n_main > 0) ok = enc(&m->group, g.sw, g.w, n_main, st ? 64 : rw, st ? 1 : 64 / rw) && enc(&m->row, g.sw, g.w, n_main, rw, 1);
    const int w0 = c.n1 > 0 ? g.w - c.n1 : 0;           // token column of the first column behind the seam
    const int n_wrapped = (c.last >= 0 ? c.last : g.Mw) - c.first_wrapped;
    if (ok && n_wrapped > 0) ok = enc(&m->wrapped, w0, g.w, n_wrapped, rw, 1);
    if (ok && c.seam >= 0) {
        const int ew = g.W - c.seam * g.w < g.w ? g.W - c.seam * g.w : g.w;
        const int cut = st ? c.n1 % 32 : c.n1;          // slots in front of the seam of the row or strip that it cuts
        if (cut > 0) ok = enc(&m->seam_a, g.W - c.n1, c.n1, 1, cut, 1);
        if (ok && cut > 0 && cut + c.skip < rw && ew > c.n1) ok = enc(&m->seam_b, 0, ew - c.n1, 1, rw - cut - c.skip, 1);
    }
    if (ok && c.last >= 0) {
        const int col = c.last >= c.first_wrapped ? w0 + (c.last - c.first_wrapped) * g.w : c.last * g.w + g.sw;
        ok = enc(&m->last, col, g.W - c.last * g.w, 1, rw, 1);
    }
    return ok;
}

bool make_win_maps(WinStripMaps* m, const WinCols& c, const Geo& g, const void* base, int ts) {
    std::memset(m, 0, sizeof *m);
    if (!make_win_maps(static_cast<WinMaps*>(m), c, g, base, ts)) return false;
    if (c.seam < 0) return true;
    const int ew = g.W - c.seam * g.w < g.w ? g.W - c.seam * g.w : g.w, box_ch = g.d >= 64 ? 64 : 32;
    const char* b = reinterpret_cast<const char*>(base);
    return encode_win_map(&m->seam_fa, g, b + (size_t)(g.W - c.n1) * ts * 2, ts, c.n1, 1, box_ch, 32, 1) && encode_win_map(&m->seam_fb, g, b, ts, ew - c.n1, 1, box_ch, 32, 1);
}
#endif  // !TERRA_ELEM_F16

namespace {
template <int D, int RW, bool ST = false>
cudaError_t launch_onepass(const Geo& g, const OnePassPlan& pl, const void* q, const void* k, const void* v, const float* bias, const void* o,
                           const float* lse, const void* d_o, void* dq, void* dk, void* dv, float* dbias, void* workspace, int sm_count,
                           cudaStream_t stream) {
    using L = Lay<D, RW, ST>;
    unsigned char* ws = reinterpret_cast<unsigned char*>(workspace);
    Params p;
    p.g = g;
    Maps<ST> mq, mk, mv, mg;
    if (!make_win_cols(&p.cols, g) || !make_win_maps(&mq, p.cols, g, q, g.ts) || !make_win_maps(&mk, p.cols, g, k, g.ts) ||
        !make_win_maps(&mv, p.cols, g, v, g.ts) || !make_win_maps(&mg, p.cols, g, d_o, g.heads * g.d))
        return cudaErrorNotSupported;
    p.split_log2 = pl.split_log2;
    p.npad = pl.npad;
    p.rmax = pl.rmax;
    p.rl = pl.rl;
    p.part_ha = !g.ph && g.sh > 0 ? (g.H - g.sh) % g.w : 0;
    p.part_row = (g.H - g.sh) / g.w;
    if (p.part_ha == 0 || (!ST && part_tiles(p.part_ha, g.H - p.part_row * g.w < g.w ? g.H - p.part_row * g.w : g.w, RW) == 0)) p.part_row = -1;
    p.gang = pl.gang;
    p.ring = pl.ring;
    p.rotate = pl.rotate;
    p.turn_log2 = 0;
    p.events = pl.npad / (D == 128 ? 64 : 128);
    p.flags = reinterpret_cast<unsigned*>(ws + pl.off_flags);
    p.rowstat = reinterpret_cast<const float4*>(ws);
    p.bias0 = reinterpret_cast<const float*>(ws + pl.off_bias0);
    p.bias1 = reinterpret_cast<const float*>(ws + pl.off_bias1);
    p.dbias_acc = reinterpret_cast<float*>(ws + pl.off_acc);
    p.slabs = reinterpret_cast<float4*>(ws + pl.off_slabs);
    p.q = (const __nv_bfloat16*)q; p.k = (const __nv_bfloat16*)k; p.v = (const __nv_bfloat16*)v; p.d_o = (const __nv_bfloat16*)d_o;
    int block_heads = kStatHeads;
    const long long stat_chunks = (long long)g.B * g.Mh * g.Mw * (pl.npad / 64);
    while (block_heads > 1 && stat_chunks * ((g.heads + block_heads - 1) / block_heads) < 4 * kPlanSms) block_heads /= 2;
    if (g.heads <= block_heads) block_heads = kStatHeads;               // (no more blocks by it)
    const unsigned stat = (unsigned)(stat_chunks * ((g.heads + block_heads - 1) / block_heads));
    const long long table = (long long)g.heads * 2 * pl.rmax * pl.rl;
    const unsigned tblocks = (unsigned)(table / 1024 + 1 < 592 ? table / 1024 + 1 : 592);
    prof_begin("swin_bwd_onepass_prep_kernel", stream);
    const auto prep = block_heads < kStatHeads ? swin_bwd_onepass_prep_kernel<D, RW, ST, true> : swin_bwd_onepass_prep_kernel<D, RW, ST, false>;
    prep<<<stat + tblocks, 256, 0, stream>>>(g, (const __nv_bfloat16*)o, (const __nv_bfloat16*)d_o, lse, bias,
        const_cast<float4*>(p.rowstat), const_cast<float*>(p.bias0), const_cast<float*>(p.bias1), p.dbias_acc, pl.npad, pl.rmax, pl.rl, stat, block_heads, p.flags, pl.flags);
    count_launch(stream);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int ctas = sm_count < kMaxCtas ? sm_count : kMaxCtas;
    auto launch = [&](auto kernel, bool inner, long long windows, int slab0, bool overlap) {
        p.inner = inner;
        p.units = windows * g.B * g.heads << pl.split_log2;
        p.slab0 = slab0;
        p.overlap = overlap;
        cudaError_t err = prepare_kernel((const void*)kernel, L::kSmemBytes);
        if (err != cudaSuccess) return err;
        prof_begin(overlap ? "swin_bwd_onepass_kernel<masked>" : "swin_bwd_onepass_kernel", stream);
        unsigned grid = (unsigned)(p.units < ctas ? p.units : ctas);
        p.gangs = (int)grid;
        if (p.gang > 1) {
            // as many CTAs as can be on the device together, or on the part of it that the stream or the process may use: a partition that
            // the query does not see refuses the launch
            for (int most = sms_of_stream(stream, ctas);; most = (int)grid / 2) {
                const GangShape fit = fit_gangs(pl, p.units, most);
                p.gangs = fit.gangs;
                p.gang = fit.gang;
                p.rotate = fit.rotate;
                p.turn_log2 = (D == 128 ? 2 : 1) - p.rotate;      // 256 queries (rotate: 128)
                grid = (unsigned)(p.gangs * p.gang);
                err = launch_together(kernel, grid, kThreads, L::kSmemBytes, stream, p.gang > 1, p, (__nv_bfloat16*)dq, (__nv_bfloat16*)dk, (__nv_bfloat16*)dv, mq, mk, mv, mg);
                if (err != cudaErrorCooperativeLaunchTooLarge) break;
                cudaGetLastError();
            }
        } else if (overlap) {
            // needs nothing of the launch before it: its CTAs take the SMs as that one's leave them
            err = launch_dependent(kernel, grid, kThreads, L::kSmemBytes, stream, p, (__nv_bfloat16*)dq, (__nv_bfloat16*)dk, (__nv_bfloat16*)dv, mq, mk, mv, mg);
        } else {
            // (brought up beside the statistics kernel its CTAs are spread less well: 64 x 128 tokens, 8 x 64, 32 x 32 windows 211 instead of 168 us a step)
            kernel<<<grid, kThreads, L::kSmemBytes, stream>>>(p, (__nv_bfloat16*)dq, (__nv_bfloat16*)dk, (__nv_bfloat16*)dv, mq, mk, mv, mg);
            err = cudaGetLastError();
        }
        if (err == cudaSuccess) count_launch(stream);
        return err;
    };
    const long long all = (long long)g.Mh * g.Mw;
    if constexpr (D == 128 || ST) {
        p.row1 = g.Mh;
        p.col1 = g.Mw;
        e = launch(swin_bwd_onepass_kernel<D, RW, 2, ST>, true, all, 0, false);
    } else {
        // the windows in front of the first row and column that need the mask
        p.row1 = g.w == RW ? g.H / g.w : 0;
        p.col1 = g.w == RW ? g.W / g.w : 0;
        // (a row of windows that are two each needs none)
        if (!g.ph && g.sh > 0 && (g.H - g.sh) % g.w && (g.H - g.sh) / g.w < p.row1 && (!L::kTwo || part_tiles((g.H - g.sh) % g.w, g.w, RW) == 0)) p.row1 = (g.H - g.sh) / g.w;
        if (!g.pw && g.sw > 0 && (g.W - g.sw) % g.w && (g.W - g.sw) / g.w < p.col1) p.col1 = (g.W - g.sw) / g.w;
        if (p.row1 == 0 || p.col1 == 0) p.row1 = p.col1 = 0;
        const long long inner = (long long)p.row1 * p.col1;
        const long long units0 = inner * g.B * g.heads << pl.split_log2;
        const int slabs0 = (int)(units0 < ctas ? units0 : ctas);
        if (inner > 0) e = launch(swin_bwd_onepass_kernel<D, RW, 0, ST>, true, inner, 0, false);
        if (e == cudaSuccess && inner < all) e = launch(swin_bwd_onepass_kernel<D, RW, 1, ST>, false, all - inner, slabs0, inner > 0);
    }
    if (e != cudaSuccess) return e;
    const int nw = 2 * g.w - 1;
    const unsigned bias_blocks = (unsigned)((nw * nw * g.heads + 255) / 256);
    const long long sum_blocks = pl.split_log2 ? (pl.units >> pl.split_log2) * ((pl.npad * D / 4 + 255) / 256) : 0;
    prof_begin("swin_bwd_onepass_finish_kernel", stream);
    e = launch_dependent(swin_bwd_onepass_finish_kernel<D, RW>, (unsigned)(bias_blocks + sum_blocks), 256, 0, stream, g, p.dbias_acc, dbias, p.slabs,
                         (__nv_bfloat16*)dq, pl.npad, pl.rmax, pl.rl, pl.split_log2, bias_blocks);
    count_launch(stream);
    return e;
}
}  // namespace

cudaError_t launch_bwd_onepass(const Geo& g, const void* q, const void* k, const void* v, const float* bias, const void* o, const float* lse,
                               const void* d_o, void* dq, void* dk, void* dv, float* dbias, void* workspace, int sm_count, cudaStream_t stream) {
    const OnePassPlan pl = bwd_onepass_plan(g);
    auto fn = pl.strips ? (g.d == 32 ? launch_onepass<32, 32, true> : g.d == 64 ? launch_onepass<64, 32, true> : launch_onepass<128, 32, true>)
            : pl.rw == 16 ? (g.d == 64 ? launch_onepass<64, 16> : launch_onepass<128, 16>)
                          : (g.d == 32 ? launch_onepass<32, 32> : g.d == 64 ? launch_onepass<64, 32> : launch_onepass<128, 32>);
    return fn(g, pl, q, k, v, bias, o, lse, d_o, dq, dk, dv, dbias, workspace, sm_count, stream);
}

}  // namespace terra
