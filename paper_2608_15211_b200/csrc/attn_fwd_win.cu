// Forward shifted-window attention on the tcgen05 tensor cores: window sides 9 .. 128 at head dims 64 and 128, 17 .. 128 at head dim 32 (less the
// sides and, above 32, the grids that fwd_win_supported leaves to the register tiles, and the complete windows of attn_fwd_tc64.cu), any grid.
//
// A unit is a pair of 128-row query tiles of one (sample, window, head), on small grids one tile; a persistent CTA per SM walks over units and streams
// the window's keys through shared memory in chunks of 128 slots (see win_tiles.cuh: 16 or 32 slots to a window row).  Per
// half chunk of 64 keys and query tile:
//   S = Q K^T (+ E_q E_k^T, see below), 128 x 64 in TMEM;
//   the softmax warps, 32 query rows each, take the rows' 64 scores into registers, add the bias, take the maximum, raise the
//   row's reference m when the half chunk exceeds it by more than 8 octaves (rare; O and the row sum are scaled down then),
//   and write P = exp2(S scale + bias - m) over S in 16 bits; the row sum is added up in fp32 before that rounding;
//   O += P V, accumulated in TMEM.
// Masks cost the softmax threads nothing: where a window's slots differ in shift-mask label or hold no token, one more
// 16-wide step of the score product (bf16 operands in either build) adds 2^64 x -2^64 to the pairs that must not see one
// another, which leaves the range of fp32: such a score is -inf whatever the scores, the scale and the bias are.  E_q holds 2^64 at
// the query's label, E_k -2^64 at every label but the key's.  What an infinity cannot be added to, a forbidden score that is
// +inf or not a number, turns up as NaN in the maximum: the half chunk's scores then go by their labels (drop_forbidden).
// (Selects by label in every half chunk of the windows that mix them, before or after the load: 256 x 512 tokens, 12 x 64,
// 32 x 32 windows, one in eight masked, 850 -> 1000 us.)  One body serves every window: the elementwise code is what bounds
// the kernel, and two copies of it in one kernel run slower than one.
// Scores and P share six TMEM buffers (head dim 128: four), so that the products of other half chunks run under the softmax.
// Sides above 32 (ST): window rows in strips of 32 slots (win_tiles.cuh), a strip in the place of a row.  The bias table of a head (0.5 MB at side
// 128) stays in L2: a thread has the 14 entries of its next half chunk in registers before it needs them (256 x 640 tokens, 8 x 128, side 128: 13.6
// ms, with table rows staged in shared memory per 128 keys 14.4; 111 x 398, 12 x 128, side 64, on mma.sync 6.75, so 1.3 ms).  Of a window whose
// mask label changes between two tiles each part is a window (part_tiles): 13.6 -> 10.6 ms at shift 64.
//
// What bounds it: the softmax warps' chain per half chunk, two warps a scheduler: 0.87 ms for 256 x 512 tokens, 12 x 64, 32 x 32 windows, of
// which the exponentials need 0.35 (16 a clock and SM); issue slots 40 %, tensor pipe 22 %, DRAM 10 %.  Head dim 128: 7.1 ms for
// 288 x 544 tokens, 64 x 128 (exponentials 2.2 ms), tensor pipe 39 %.
//
// Roles (512 threads): warps 0-3 / 4-7 softmax of the pair's first / second tile, warps 8-11 read O out of TMEM, normalise
// and store it, warp 12 issues the PV products, warp 13 every copy, warp 14 the scores, warp 15 walks over the units.
// Every mbarrier wait is bounded; on expiry the CTA raises an abort flag, all roles leave their loops, TMEM is released and
// the host reads the device status word.
#include "swin_common.cuh"
#include "swin_kernels.h"
#include "tc_common.cuh"
#include "win_tiles.cuh"

// fp16 build of this file (through the _f16 wrapper file): names of its own
#ifdef TERRA_ELEM_F16
#define g_fwd_win_timeout g_fwd_win_timeout_f16
#define launch_fwd_win launch_fwd_win_f16
#define read_fwd_win_status read_fwd_win_status_f16
#endif

namespace terra {

__device__ int g_fwd_win_timeout = 0;   // set when a bounded wait expired in any CTA of the kernel below

namespace {

using namespace tc;

constexpr int kThreads = 512;
constexpr int kSoftWarps = 8, kReadWarp0 = 8, kPvWarp = 12, kLoaderWarp = 13, kScoreWarp = 14, kPlanWarp = 15;
constexpr int kRegsLaunch = 128, kRegsSoft = 184, kRegsOther = 72;
static_assert(2 * kRegsSoft + 2 * kRegsOther <= 4 * kRegsLaunch, "register hand-over does not balance");
constexpr int kTile = 128, kDescs = 8;
constexpr uint32_t kMaskQ = 0x5F80, kMaskK = 0xDF80;           // bf16 2^64, -2^64
constexpr float kLowest = -3.402823466e38f;                    // a row's reference before its first key

// The bias table by row difference, twice: copy c starts at column difference c - (RW - 1), so that a thread's pairs of keys
// are read aligned, from the copy of its row's parity; the copies lie 16 banks apart.
template <int RW>
struct Tab {
    static constexpr int kCopyF = RW == 16 ? 48 : 80, kRowF = 2 * kCopyF;
    static constexpr int kFront = RW == 16;                   // a row in front of the first difference: two query rows share their reads
    static __host__ __device__ constexpr int rows(int w) { return 2 * w + 2 * kFront; }
};

// Full barriers: a slot has one for its Q and K tiles (the score warp waits for each of them) and one for its V tiles (the product warp).
// A wait names a phase by parity, so nobody may skip a fill of a barrier he waits on: with one barrier for both, a V tile that was
// later than the scores let the next unit's first scores pass their wait for the K tile that goes to the same slot (head dim 128,
// 32 x 32 windows: one call in a thousand).  (Waiting for V in the score warp as well: 240 x 360 tokens, 6 x 64, side 18 396 us; so 358.)
enum { kBFull = 0, kBEmpty = 16, kBS = 32, kBP = 38, kBFree = 44, kBO = 50, kBOFree = 52, kBStat = 54, kBTab = 56, kBBias = 58,
       kBOne = 59, kBDesc = 61, kBDescFree = kBDesc + kDescs, kBFullV = kBDescFree + kDescs, kBCount = kBFullV + 16 };

template <int D, int RW, bool ST>
struct Lay {
    static constexpr int kParts = D == 128 ? 2 : 1, kRowB = D >= 64 ? 128 : 64, kPartCh = kRowB / 2;
    static constexpr int kSlotB = kTile * D * 2;                                    // a Q, K or V tile
    static constexpr int kSlots = D == 128 ? (RW == 16 ? 6 : 5) : D == 64 ? 10 : 14;
    static constexpr int kBufs = D == 128 ? 4 : 6, kColO = 64 * kBufs;
    static constexpr int kOffE = kSlots * kSlotB;                                   // E operands, 64 bytes a slot: E_q, then E_k
    static constexpr int kEUnits = ST ? 12 : 256 / RW;                              // rows of slots (ST: strips) of the E operands
    static constexpr int kOffTab = kOffE + kEUnits * RW * 64;
    static constexpr int kOffStat = kOffTab + (ST ? 0 : Tab<RW>::rows(RW) * Tab<RW>::kRowF * 4);          // per row of both tiles: m, row sum
    static constexpr int kOffDesc = kOffStat + 2 * kTile * 8;
    static constexpr int kOffBars = kOffDesc + kDescs * 64;
    static constexpr int kSmemBytes = kOffBars + 8 * kBCount + 16;
};

struct Params {
    Geo g;
    WinCols cols;
    const __nv_bfloat16 *q, *k, *v;
    const float* tables;         // [head][Tab::rows][Tab::kRowF]; ST: [head][2 w - 1][2][64 strips], read from global memory
    int strips;                  // ST: strips of a full window row
    int tiles;                   // query tiles of a unit: 2, or 1 where that leaves every unit a CTA
    int units_win, units_row;    // units of a window of full height, and of one of the last, truncated window row
    int rows;                    // window rows of full height
    int part_row, part_ha;       // the window row whose windows may be two parts, -1: none (see part_tiles), and the second part's first row
    int head_slow;               // units in head-major order, a run per CTA; else the head is the fastest digit, strided
    long long units;
};

struct Unit {
    int head, b, wr, wc;
    int eh, ew, tile0, ntq;      // first query tile, 1 or 2 of them
    int ku, nch, ha, hb;         // 32-slot key units, chunks; window rows >= ha / columns >= hb carry the other mask label
    int flags;                   // 1: a unit (0: the end), 2: another head than before, 4: the scores need the mask step
    int ns;                      // ST: strips of a window row
    int c0;                      // first chunk of keys
};

// ST: rows of strips per row label among the mask operands, so that four strips in a row from any strip on lie in them
__device__ __forceinline__ int e_rows(int ns) { return ns == 1 ? 4 : ns == 4 ? 1 : 2; }

template <bool ST>
using Maps = std::conditional_t<ST, WinStripMaps, WinMaps>;

// FIFO of shared-memory slots: two held for a unit (Q tiles), the others cycle (K, V chunks)
template <int N>
struct SlotQueue {
    uint64_t q;
    __device__ __forceinline__ void init() {
        q = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) q |= (uint64_t)i << (4 * i);
    }
    __device__ __forceinline__ int pop() { const int s = (int)(q & 15); q >>= 4; return s; }
    __device__ __forceinline__ int take() { const int s = pop(); q |= (uint64_t)s << (4 * (N - 3)); return s; }
    __device__ __forceinline__ void end_unit(int s0, int s1) { q |= ((uint64_t)s0 << (4 * (N - 2))) | ((uint64_t)s1 << (4 * (N - 1))); }
};

__device__ __forceinline__ float2 lds_f2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}

__device__ __forceinline__ float max3_nan(float a, float b, float c) {
    float d;
    asm("max.NaN.f32 %0, %1, %2, %3;\n" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// The thread's scores of one 32-slot key unit (32 query rows x 32 keys a warp; thread 4 g + t holds rows g + 8 m, keys
// 8 k + 2 t + e) -> S scale + bias in place, and the rows' maxima (NaN if a score is).  Pairs on one diagonal share their bias: 7 or 9 reads
// for 32 scores.  (A thread per row read each score's own entry: the shared-memory pipe then bound the kernel, 1300 to 2500
// of 4100 to 6800 cycles per 128 x 128 scores and tile.)  `bias`: shared address of the entry of rows g, keys 2 t.
template <int RW>
__device__ __forceinline__ void load_bias(float2 (&bv)[RW == 32 ? 7 : 9], uint32_t bias) {
    constexpr int kRowB = Tab<RW>::kRowF * 4;
#pragma unroll
    for (int i = 0; i < (RW == 32 ? 7 : 9); ++i)
        bv[i] = lds_f2(bias + (RW == 32 ? 32 * (i - 3) : (i / 3 - 1) * kRowB + 32 * (i % 3 - 1)));
}
template <int RW, int KC>
__device__ __forceinline__ void add_bias(uint32_t (&x)[2][32], int u, const float2 (&bv)[RW == 32 ? 7 : 9], float scale, float (&mx)[4]) {
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int k = 0; k < KC; ++k) {
            uint32_t* v = &x[m >> 1][16 * u + 4 * k + 2 * (m & 1)];
            const float2 b = bv[RW == 32 ? k - m + 3 : 3 * ((k >> 1) - (m >> 1) + 1) + (k & 1) - (m & 1) + 1];
            float x0, x1;
            fma2(x0, x1, __uint_as_float(v[0]), __uint_as_float(v[1]), scale, b.x, b.y);
            v[0] = __float_as_uint(x0);
            v[1] = __float_as_uint(x1);
            mx[m] = max3_nan(mx[m], x0, x1);
        }
}

// The scores of a half chunk (key rows `ak` on, `cols` of its columns; 32 query rows a warp, window row `aq` on) whose tokens differ in
// mask label become -inf, in tensor memory.  Not inlined, and the half chunk starts over from the loop's head: with this code in the
// middle of the softmax's every unit paid for it (121 x 250 x 2 tokens, 8 x 64, side 32: 285 -> 306 us; so 290).
// ST: `ak` and `aq` are units, `ns` to a window row.
template <int RW, bool ST>
__device__ __noinline__ void drop_forbidden(uint32_t t_s, int cols, int ak, int aq, int ha, int hb, int gl, int ql, int ns) {
#pragma unroll 1
    for (int c = 0; c < cols; c += 16)
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            // 16 keys x 16 queries, each of one window row
            const int uk = ak + c / RW, uq = aq + (RW == 32 ? 0 : h), rk = ST ? unit_row(uk, ns) : uk, rq = ST ? unit_row(uq, ns) : uq;
            const bool rows = (rk >= ha) == (rq >= ha);
            const int ck = ST ? 32 * (uk - rk * ns) : 0, cq = ST ? 32 * (uq - rq * ns) : 0;
            uint32_t r[8];
            tmem_ld_frag16(t_s + ((16u * h) << 16) + c, r);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int bk = ck + (RW == 32 ? c & 16 : 0) + 8 * (i >> 2) + 2 * ql + (i & 1), bq = cq + (RW == 32 ? 16 * h : 0) + 8 * ((i >> 1) & 1) + gl;
                r[i] = rows && (bk >= hb) == (bq >= hb) ? r[i] : 0xff800000u;
            }
            tmem_st_frag16(t_s + ((16u * h) << 16) + c, r);
        }
    tmem_st_wait();
}

// KC: of every 32 key slots the first 8 KC are worked on (window sides 17 .. 24 in rows of 32 slots leave the last 8 without a
// token: 3; otherwise 4).  240 x 360 tokens, 6 x 64, side 22: 357 -> 302 us.
// TWO: windows of two parts (part_tiles) as such.  Of its own below side 33: the code for it cost grids without such windows 1 to 5 % (108 x 230 tokens,
// 30 x 128, side 9 685 us, so 648; 2 x 299 x 796, 2 x 64, side 13 333, so 327; 2 x 299 x 796, 2 x 128, side 12 499, so 479).
template <int D, int RW, int KC, bool ST, bool TWO>
__global__ void __launch_bounds__(kThreads, 1)
swin_fwd_win_kernel(const __grid_constant__ Params p, __nv_bfloat16* __restrict__ o, float* __restrict__ lse,
                    const __grid_constant__ Maps<ST> mq, const __grid_constant__ Maps<ST> mk, const __grid_constant__ Maps<ST> mv) {
    using L = Lay<D, RW, ST>;
    constexpr int kParts = L::kParts, kRowB = L::kRowB, kG = 64 / RW, NB = L::kBufs, kTileRows = kTile / RW;
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
            mbar_init(bar(kBFullV + s), 1);
            mbar_init(bar(kBEmpty + s), 1);
        }
        for (int b = 0; b < NB; ++b) {
            mbar_init(bar(kBS + b), 1);            // scores of a half chunk are in buffer b
            mbar_init(bar(kBP + b), 4);            // ... and P has taken their place
            mbar_init(bar(kBFree + b), 1);         // ... and been read by the product
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(bar(kBO + t), 1);            // ... the unit's last one
            mbar_init(bar(kBOFree + t), 4);        // O and the statistics of tile t have been read
            mbar_init(bar(kBStat + t), 4);         // the rows' m and sums are in shared memory
            mbar_init(bar(kBTab + t), kSoftWarps); // the softmax of a unit is done (even / odd units)
            mbar_init(bar(kBOne + t), 4);          // ... of a unit of one tile (even / odd ones): the other warps keep in step
        }
        mbar_init(bar(kBBias), 1);                 // the head's bias table is in shared memory
        for (int i = 0; i < kDescs; ++i) {
            mbar_init(bar(kBDesc + i), 1);
            mbar_init(bar(kBDescFree + i), kSoftWarps + 7);
        }
        *cta_abort = 0;
        fence_barrier_init();
    }
    if (warp == kPvWarp) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    wait_for_prerequisites();                      // the bias tables
    unsigned desc_n = 0;
    Unit td;
    // the next unit; false at the end of the run (or after an expired wait)
    auto next_unit = [&]() {
        const unsigned i = desc_n % kDescs;
        if (!mbar_wait_all(bar(kBDesc + i), (desc_n / kDescs) & 1, cta_abort)) return false;
        const int4* src = reinterpret_cast<const int4*>(smem + L::kOffDesc + i * 64);
        const int4 d0 = src[0], d1 = src[1], d2 = src[2];
        td.head = d0.x; td.b = d0.y; td.wr = d0.z; td.wc = d0.w;
        td.eh = d1.x; td.ew = d1.y; td.tile0 = d1.z; td.ntq = d1.w;
        td.ku = d2.x; td.nch = d2.y; td.ha = d2.z; td.hb = d2.w;
        const int4 d3 = src[3];
        td.flags = d3.x; td.c0 = TWO ? d3.z : 0;
        if (ST) td.ns = d3.y;
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(kBDescFree + i));
        ++desc_n;
        return (td.flags & 1) != 0;
    };

    if (warp < kSoftWarps) {
        // ------------------------------------------------------------------ softmax of tile t
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kRegsSoft));
        const int t = warp >> 2, wq = warp & 3, gl = lane >> 2, ql = lane & 3;
        const uint32_t tq = tmem + ((uint32_t)(32 * wq) << 16), t_o = tq + L::kColO + D * t;
        const float scale = g.scale_log2e;
        const int i0 = RW - 1 + 2 * ql - gl;                 // table column of row g, key 2 t
        const uint32_t tab0 = smem0 + L::kOffTab + 4u * ((i0 & 1) * Tab<RW>::kCopyF + (i0 & ~1));
        float2* stat = reinterpret_cast<float2*>(smem + L::kOffStat) + t * kTile + 32 * wq + gl;
        unsigned n = 0, units = 0, mine = 0, heads = 0, ones = 0;   // half chunks of the CTA; units, those with this tile; tables; 1-tile units
        bool ok = true;
        while (ok && next_unit()) {
            if (!ST && (td.flags & 2)) ok = mbar_wait_all(bar(kBBias), heads++ & 1, cta_abort);
            if (ok && t < td.ntq) {
                const int aq = min((td.tile0 + t) * kTileRows + wq * (32 / RW), (ST ? td.ku : td.eh) - 1);
                uint32_t bias = tab0 + 4u * (g.w - 1 - aq + Tab<RW>::kFront + td.c0 * kTileRows) * Tab<RW>::kRowF;
                // ST: the entries of the next half chunk's two key units, from the head's table in L2, are in registers before they are needed
                float2 bv[ST ? 2 : 1][RW == 32 ? 7 : 9];
                const float* bp = nullptr;
                int sk = 0;
                auto next_bias = [&](int left) {             // key units left
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (u < left) {
#pragma unroll
                            for (int i = 0; i < 7; ++i) bv[ST ? u : 0][i] = __ldg(reinterpret_cast<const float2*>(bp + 8 * (i - 3)));
                        }
                        bp += 32;
                        if (++sk == td.ns) { sk = 0; bp += 128 * p.strips - 32 * td.ns; }
                    }
                };
                if (ST) {
                    const int rq = unit_row(aq, td.ns), j0 = 32 * p.strips - 1 + 2 * ql - gl;
                    bp = p.tables + ((size_t)td.head * (2 * g.w - 1) + g.w - 1 - rq) * (128 * p.strips) + (j0 & 1) * (64 * p.strips) + (j0 & ~1) - 32 * (aq - rq * td.ns);
                    const int rk = unit_row(4 * td.c0, td.ns);
                    sk = 4 * td.c0 - rk * td.ns;
                    bp += rk * 128 * p.strips + 32 * sk;
                    next_bias(td.ku - 4 * td.c0);
                }
                float m[4] = {kLowest, kLowest, kLowest, kLowest};     // (finite: a half chunk may hold no key that the row sees)
                float2 sum[4] = {};
                int fixed = -1;                          // half chunk whose scores have gone by their labels
                const int j0 = 2 * td.c0;
                for (int j = j0; 2 * j < td.ku; ++j) {
                    const unsigned idx = n + (j - j0) * td.ntq + t, buf = idx % NB;
                    const uint32_t t_s = tq + 64u * buf;
                    ok = mbar_wait_all(bar(kBS + buf), (idx / NB) & 1, cta_abort);
                    if (!ok) break;
                    tc_fence_after();
                    uint32_t x[2][32];                       // [rows g + 16 h, + 8]
                    tmem_ld_frag64(t_s, x[0]);
                    tmem_ld_frag64(t_s + (16u << 16), x[1]);
                    tmem_ld_wait();
                    float top[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                    if (!ST) load_bias<RW>(bv[0], bias);
                    add_bias<RW, KC>(x, 0, bv[0], scale, top);
                    if (2 * j + 1 < td.ku) {
                        if (!ST) load_bias<RW>(bv[0], bias + 4u * (32 / RW) * Tab<RW>::kRowF);
                        add_bias<RW, KC>(x, 1, bv[ST ? 1 : 0], scale, top);
                    } else {
                        // 32 slots that do not exist
#pragma unroll
                        for (int i = 16; i < 32; ++i) x[0][i] = x[1][i] = 0xff800000u;
                    }
                    if (!__all_sync(0xffffffffu, top[0] - m[0] <= 8.f && top[1] - m[1] <= 8.f && top[2] - m[2] <= 8.f && top[3] - m[3] <= 8.f)) {
                        if (fixed != j && ((td.ha > 0 && td.ha < td.eh) || (td.hb > 0 && td.hb < td.ew)) &&
                            __any_sync(0xffffffffu, top[0] != top[0] || top[1] != top[1] || top[2] != top[2] || top[3] != top[3])) {
                            drop_forbidden<RW, ST>(t_s, 32 * min(2, td.ku - 2 * j), 2 * j * (32 / RW), (td.tile0 + t) * kTileRows + wq * (32 / RW), td.ha, td.hb, gl, ql, ST ? td.ns : 1);
                            fixed = j--;
                            continue;
                        }
                        // raise the reference; O and the sums so far are scaled down, once the products so far are done
                        float f[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            top[i] = fmaxf(top[i], __shfl_xor_sync(0xffffffffu, top[i], 1));
                            top[i] = fmaxf(top[i], __shfl_xor_sync(0xffffffffu, top[i], 2));
                            const float up = top[i] - m[i] > 8.f ? top[i] : m[i];
                            f[i] = fast_exp2(m[i] - up);
                            m[i] = up;
                            sum[i].x *= f[i];
                            sum[i].y *= f[i];
                        }
                        if (j > j0) {
                            // (the buffer of the last product cannot be freed again before this half chunk's product)
                            const unsigned last = idx - td.ntq;
                            ok = mbar_wait_all(bar(kBFree + last % NB), (last / NB) & 1, cta_abort);
                            if (!ok) break;
                            tc_fence_after();
#pragma unroll 1
                            for (int col = 0; col < D; col += 16)
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    uint32_t r[8];
                                    tmem_ld_frag16(t_o + ((16u * h) << 16) + col, r);
                                    tmem_ld_wait();
#pragma unroll
                                    for (int i = 0; i < 8; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * f[2 * h + ((i >> 1) & 1)]);
                                    tmem_st_frag16(t_o + ((16u * h) << 16) + col, r);
                                }
                        }
                    }
                    if (ST && 2 * (j + 1) < td.ku) next_bias(td.ku - 2 * (j + 1));
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        uint32_t pk[16];
#pragma unroll
                        for (int k = 0; k < 8; ++k)
#pragma unroll
                            for (int mi = 0; mi < 2; ++mi) {
                                const int i = 2 * h + mi;
                                if ((k & 3) >= KC) {
                                    pk[2 * k + mi] = 0u;
                                    continue;
                                }
                                float x0, x1;
                                add2(x0, x1, __uint_as_float(x[h][4 * k + 2 * mi]), __uint_as_float(x[h][4 * k + 2 * mi + 1]), -m[i]);
                                x0 = fast_exp2(x0);
                                x1 = fast_exp2(x1);
                                add2vv(sum[i].x, sum[i].y, sum[i].x, sum[i].y, x0, x1);
                                pk[2 * k + mi] = pack_elem(x0, x1);
                            }
                        tmem_st_frag_packed32(t_s + ((16u * h) << 16), pk);
                    }
                    bias += 4u * (64 / RW) * Tab<RW>::kRowF;
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kBP + buf));
                }
                if (ok) {
                    // the last unit's statistics have been read
                    ok = mbar_wait_all(bar(kBOFree + t), (mine & 1) ^ 1u, cta_abort);
                    ++mine;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float s = sum[i].x + sum[i].y;
                        s += __shfl_xor_sync(0xffffffffu, s, 1);
                        s += __shfl_xor_sync(0xffffffffu, s, 2);
                        if (ql == 0) stat[8 * i] = make_float2(m[i], s);
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(kBStat + t));
                }
            }
            if (td.ntq == 1) {
                // barriers are waited for by parity: warps that skip units must not be ahead of the scores or the tables
                if (t == 0) {
                    if (lane == 0) mbar_arrive(bar(kBOne + (ones & 1)));
                } else {
                    ok = ok && mbar_wait_all(bar(kBOne + (ones & 1)), (ones >> 1) & 1, cta_abort);
                }
                ++ones;
            }
            if (lane == 0) mbar_arrive(bar(kBTab + (units & 1)));
            ++units;
            n += (((td.ku + 1) >> 1) - 2 * td.c0) * td.ntq;
        }
    } else if (warp < kPvWarp) {
        // ------------------------------------------------------------------ O: normalise and store
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kRegsOther));
        const int wq = warp - kReadWarp0, row = 32 * wq + lane;
        const uint32_t t_o = tmem + ((uint32_t)(32 * wq) << 16) + L::kColO;
        unsigned done[2] = {0, 0};
        bool ok = true;
        while (ok && next_unit()) {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                if (t >= td.ntq) break;
                const int slot = (td.tile0 + t) * kTile + row, ua = slot / RW, a = ST ? unit_row(ua, td.ns) : ua, bb = slot % RW + (ST ? 32 * (ua - a * td.ns) : 0);
                ok = mbar_wait_all(bar(kBStat + t), done[t] & 1, cta_abort) && mbar_wait_all(bar(kBO + t), done[t] & 1, cta_abort);
                if (!ok) break;
                ++done[t];
                tc_fence_after();
                const float2 st = reinterpret_cast<const float2*>(smem + L::kOffStat)[t * kTile + row];
                const float inv = 1.f / st.y;
                const bool live = a < td.eh && bb < td.ew;
                const size_t tok = live ? (size_t)td.b * g.H * g.W + win_token(g, td.wr, td.wc, a, bb) : 0;
                uint4* dst = reinterpret_cast<uint4*>(o + (tok * g.heads + td.head) * D);
#pragma unroll
                for (int col = 0; col < D; col += 32) {
                    uint32_t r[32];
                    tmem_ld32(t_o + D * t + col, r);
                    tmem_ld_wait();
                    if (col + 32 == D) {
                        // all of it is in registers
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar(kBOFree + t));
                    }
                    if (live) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            uint32_t w[4];
#pragma unroll
                            for (int j = 0; j < 4; ++j) w[j] = pack_elem(__uint_as_float(r[8 * i + 2 * j]) * inv, __uint_as_float(r[8 * i + 2 * j + 1]) * inv);
                            dst[col / 8 + i] = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                }
                if (live) lse[tok * g.heads + td.head] = (st.x + log2f(st.y)) * kLn2;
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kRegsOther));
        if (warp == kPlanWarp) {
            // -------------------------------------------------------------- units in the order every role meets them
            unsigned i = 0;
            int last_head = -1;
            bool ok = true;
            auto put = [&](int flags, int head, int b, int wr, int wc, int eh, int ew, int tile0, int t0) {
                ok = mbar_wait_all(bar(kBDescFree + i % kDescs), ((i / kDescs) & 1) ^ 1u, cta_abort);
                if (!ok) return;
                if (lane == 0) {
                    const int ha = (!g.ph && g.sh > 0) ? g.H - g.sh - wr * g.w : (1 << 20), hb = (!g.pw && g.sw > 0) ? g.W - g.sw - wc * g.w : (1 << 20);
                    const int ns = ST ? strips_of(ew) : 1, nqt = (eh * ns * RW + kTile - 1) / kTile, ku_all = RW == 32 ? eh * ns : (eh + 1) / 2;
                    // a window of two parts: the part's keys (t0: the second part's first tile)
                    const int c0 = t0 > 0 && tile0 >= t0 ? t0 : 0, ku = t0 > 0 && tile0 < t0 ? 4 * t0 : ku_all;
                    if (ew < ns * RW || (ha > 0 && ha < eh && t0 == 0) || (hb > 0 && hb < ew) || (RW == 16 && (eh & 1))) flags |= 4;
                    int4* dst = reinterpret_cast<int4*>(smem + L::kOffDesc + (i % kDescs) * 64);
                    dst[0] = make_int4(head, b, wr, wc);
                    dst[1] = make_int4(eh, ew, tile0, min(p.tiles, nqt - tile0));
                    dst[2] = make_int4(ku, (ku + 3) / 4, ha, hb);
                    dst[3] = make_int4(flags, ns, c0, 0);
                    mbar_arrive(bar(kBDesc + i % kDescs));
                }
                __syncwarp();
                ++i;
            };
            const long long lo = p.head_slow ? p.units * blockIdx.x / gridDim.x : blockIdx.x, hi = p.head_slow ? p.units * (blockIdx.x + 1) / gridDim.x : p.units;
            const int step = p.head_slow ? 1 : gridDim.x;
            const unsigned per_head = (unsigned)(p.units / g.heads);
            for (long long u = lo; ok && u < hi; u += step) {
                unsigned rest, head;
                if (p.head_slow) { head = (unsigned)u / per_head; rest = (unsigned)u - head * per_head; }
                else { rest = (unsigned)u / g.heads; head = (unsigned)u - rest * g.heads; }
                // sample, then the windows of full height, then the last row's
                const unsigned full = (unsigned)p.rows * g.Mw * p.units_win, per_sample = full + (unsigned)(g.Mh - p.rows) * g.Mw * p.units_row;
                const unsigned b = rest / per_sample, in = rest - b * per_sample, each = in < full ? p.units_win : p.units_row, at = in < full ? in : in - full;
                const unsigned win = at / each, unit = at - win * each, row = win / g.Mw, wc = win - row * g.Mw, wr = in < full ? row : p.rows;
                const int eh = min(g.w, g.H - (int)wr * g.w), ew = min(g.w, g.W - (int)wc * g.w);
                if (ST && (int)unit * p.tiles * kTileRows >= eh * strips_of(ew)) continue;            // a truncated window has fewer query tiles
                // (not where a pair of tiles would be of either part: one after the other, 288 x 544 tokens, 8 x 128, side 16, took 341 us; as one window 300)
                int t0 = !TWO || (int)wr != p.part_row ? 0 : part_tiles(p.part_ha, eh, (ST ? strips_of(ew) : 1) * RW);
                if (t0 & (p.tiles - 1)) t0 = 0;
                put(1 | ((int)head != last_head ? 2 : 0), head, b, wr, wc, eh, ew, unit * p.tiles, t0);
                last_head = head;
            }
            if (ok) put(0, 0, 0, 0, 0, 1, 1, 0, 0);
        } else if (warp == kLoaderWarp) {
            // -------------------------------------------------------------- copies, bias tables, mask operands
            SlotQueue<L::kSlots> sq;
            sq.init();
            uint32_t use = 0;                        // bit per slot: parity of the slot's fills
            unsigned units = 0;
            int e_key = -1, q0 = -1, q1 = -1;        // what the mask operands are made for; Q slots of the last unit
            bool ok = true;
            const int part = lane % kParts, row = lane / kParts;      // lane -> channel part, window row of a tile
            // ST: of the tile's four strips from `a0` on those that the seam cuts
            auto cut_units = [&](int a0) {
                int n = 0;
                for (int u = a0; u < a0 + 4; ++u) n += u - unit_row(u, td.ns) * td.ns == p.cols.n1 >> 5;
                return n;
            };
            auto fill = [&](int s, int full, const Maps<ST>& m, const __nv_bfloat16* src, int a0) {
                ok = ok && mbar_wait_all(bar(kBEmpty + s), ((use >> s) & 1) ^ 1u, cta_abort);
                if (!ok) return;
                use ^= 1u << s;
                const bool fix = D == 32 && p.cols.skip && td.wc == p.cols.seam;
                if (D == 32 && fix) {
                    // the seam column's slot n1 cannot be the start of a bulk copy of 64-byte rows (128-byte alignment)
                    for (int i = lane; i < 2 * kG * 4; i += 32) {
                        const int r = i >> 2, ch = i & 3, a = ST ? unit_row(a0 + r, td.ns) : a0 + r, cut = ST ? p.cols.n1 & 31 : p.cols.n1;
                        if (ST && a0 + r - a * td.ns != p.cols.n1 >> 5) continue;
                        uint4 val = make_uint4(0, 0, 0, 0);
                        if (a < td.eh && p.cols.n1 < td.ew)
                            val = __ldg(reinterpret_cast<const uint4*>(src + ((size_t)td.b * g.H * g.W + win_token(g, td.wr, td.wc, a, p.cols.n1)) * g.ts + td.head * D) + ch);
                        *reinterpret_cast<uint4*>(smem + s * L::kSlotB + tile_off<32>(r * RW + cut, ch)) = val;
                    }
                    fence_proxy_async();
                    __syncwarp();
                }
                const uint32_t base = smem0 + s * L::kSlotB;
                if constexpr (ST) {
                    // 64 slots of a window row are one copy where the strips are even in number, a strip one where they are not
                    const bool two = (td.ns & 1) == 0 && td.wc != p.cols.seam && td.wc < p.cols.first_wrapped && td.wc != p.cols.last;
                    if (lane == 0) mbar_arrive_expect_tx(bar(full + s), L::kSlotB - (fix ? cut_units(a0) * kRowB : 0));
                    __syncwarp();
                    if (row < (two ? 2 : 4)) {
                        const int u = a0 + (two ? 2 : 1) * row, a = unit_row(u, td.ns), st = u - a * td.ns;
                        const uint32_t dst = base + part * kTile * kRowB + (u - a0) * 32 * kRowB;
                        if (two) {
                            int y = td.wr * g.w + a + g.sh;
                            if (y >= g.H) y -= g.H;
                            tma_load_4d(dst, &m.group, td.head * D + part * L::kPartCh, 32 * st, td.wc, a < td.eh ? td.b * g.H + y : g.B * g.H, bar(full + s));
                        } else {
                            load_win_strip<kRowB>(m, p.cols, dst, g, td.b, td.wr, td.wc, td.eh, a, st, td.head * D + part * L::kPartCh, bar(full + s));
                        }
                    }
                } else if (win_group_whole<RW>(p.cols, g, td.wr, td.wc, td.eh, a0, 2)) {
                    if (elect_one()) {
                        mbar_arrive_expect_tx(bar(full + s), L::kSlotB);
                        int y0 = td.wr * g.w + a0 + g.sh;
                        if (y0 >= g.H) y0 -= g.H;
                        y0 += td.b * g.H;
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int pt = 0; pt < kParts; ++pt)
                                tma_load_4d(base + pt * kTile * kRowB + h * 64 * kRowB, &m.group, td.head * D + pt * L::kPartCh, 0, td.wc, y0 + h * kG, bar(full + s));
                    }
                } else {
                    if (lane == 0) mbar_arrive_expect_tx(bar(full + s), L::kSlotB - (fix ? 2 * kG * kRowB : 0));
                    __syncwarp();
                    if (row < 2 * kG)
                        load_win_row<RW, kRowB>(m, p.cols, base + part * kTile * kRowB + row * RW * kRowB, g, td.b, td.wr, td.wc, td.eh, a0 + row,
                                                td.head * D + part * L::kPartCh, bar(full + s));
                }
                __syncwarp();
            };
            while (ok && next_unit()) {
                // at most two units ahead of the softmax: the barriers of even and odd units are waited for once per use
                if (units >= 2) ok = mbar_wait_all(bar(kBTab + (units & 1)), ((units - 2) >> 1) & 1, cta_abort);
                if (!ST && ok && (td.flags & 2)) {
                    if (units >= 1) ok = mbar_wait_all(bar(kBTab + ((units - 1) & 1)), ((units - 1) >> 1) & 1, cta_abort);
                    if (ok && elect_one()) {
                        const uint32_t bytes = Tab<RW>::rows(g.w) * Tab<RW>::kRowF * 4;
                        mbar_arrive_expect_tx(bar(kBBias), bytes);
                        bulk_load(smem0 + L::kOffTab, p.tables + (size_t)td.head * Tab<RW>::rows(g.w) * Tab<RW>::kRowF, bytes, bar(kBBias));
                    }
                    __syncwarp();
                }
                if (ok && (td.flags & 4)) {
                    // 32 slots to a row: rows 0-3 carry the first row label, 4-7 the second; a tile starts where its rows change
                    // ST: e_rows(ns) rows of strips carry the first row label, as many the second
                    const int ha = min(max(td.ha, 0), td.eh), hb = min(max(td.hb, 0), td.ew);
                    const int key = ST ? td.ew | hb << 8 : RW == 32 ? td.ew | hb << 6 : td.ew | hb << 6 | td.eh << 12 | ha << 18;
                    if (key != e_key) {
                        e_key = key;
                        // the last unit's scores are done when its Q slots are free
                        if (q0 >= 0) ok = ok && mbar_wait_all(bar(kBEmpty + q0), ((use >> q0) & 1) ^ 1u, cta_abort);
                        if (q1 >= 0) ok = ok && mbar_wait_all(bar(kBEmpty + q1), ((use >> q1) & 1) ^ 1u, cta_abort);
                        if (ok) {
                            for (int s = lane; s < L::kEUnits * RW; s += 32) {
                                const int u = s / RW, a = ST ? unit_row(u, td.ns) : u, b = s % RW + (ST ? 32 * (u - a * td.ns) : 0);
                                const bool valid = b < td.ew && (RW == 32 || a < td.eh);
                                const int label = 2 * (RW == 32 ? a >= (ST ? e_rows(td.ns) : 4) : a >= ha) + (b >= hb);
                                uint32_t eq[2] = {0, 0}, ek[2] = {kMaskK | kMaskK << 16, kMaskK | kMaskK << 16};
                                if (valid) {
                                    const uint32_t half = (label & 1) ? 0xffff0000u : 0xffffu;
#pragma unroll
                                    for (int i = 0; i < 2; ++i)
                                        if (i == label >> 1) { eq[i] = (kMaskQ | kMaskQ << 16) & half; ek[i] &= ~half; }
                                }
                                unsigned char* e = smem + L::kOffE;
                                *reinterpret_cast<uint4*>(e + tile_off<32>(s, 0)) = make_uint4(eq[0], eq[1], 0, 0);
                                *reinterpret_cast<uint4*>(e + tile_off<32>(s, 1)) = make_uint4(0, 0, 0, 0);
                                *reinterpret_cast<uint4*>(e + tile_off<32>(s, 2)) = make_uint4(ek[0], ek[1], 0, 0);
                                *reinterpret_cast<uint4*>(e + tile_off<32>(s, 3)) = make_uint4(0, 0, 0, 0);
                            }
                            fence_proxy_async();
                            __syncwarp();
                        }
                    }
                }
                q0 = sq.pop();
                q1 = sq.pop();
                fill(q0, kBFull, mq, p.q, td.tile0 * kTileRows);
                for (int c = td.c0; ok && c < td.nch; ++c) {
                    fill(sq.take(), kBFull, mk, p.k, c * kTileRows);
                    if (c == td.c0 && td.ntq == 2) fill(q1, kBFull, mq, p.q, (td.tile0 + 1) * kTileRows);
                    fill(sq.take(), kBFullV, mv, p.v, c * kTileRows);
                }
                sq.end_unit(q0, q1);
                if (td.ntq < 2) q1 = -1;
                ++units;
            }
        } else if (warp == kScoreWarp) {
            // -------------------------------------------------------------- S = Q K^T
            constexpr uint32_t kIdS = make_idesc_elem(128, 0, 0, 0), kIdE = make_idesc_bf16(128, 0, 0, 0);
            const uint64_t d_k = D == 32 ? make_sdesc_sw64(smem0, 512) : make_sdesc_sw128(smem0);
            const uint64_t d_e = make_sdesc_sw64(smem0 + L::kOffE, 512);
            const uint32_t hi = sdesc_hi(d_k), lo = sdesc_lo(d_k), hi_e = sdesc_hi(d_e), lo_e = sdesc_lo(d_e);
            constexpr int kPerPart = L::kPartCh / 16;
            SlotQueue<L::kSlots> sq;
            sq.init();
            uint32_t full_use = 0;
            unsigned idx = 0;
            bool ok = true;
            auto wait_full = [&](int s) {
                ok = ok && mbar_wait_all(bar(kBFull + s), (full_use >> s) & 1, cta_abort);
                full_use ^= 1u << s;
            };
            // where the rows from window row a0 on start among the mask operands (16-byte units)
            auto mask_rows = [&](int a0) {
                if (ST) {
                    const int a = unit_row(a0, td.ns);
                    return (uint32_t)(min(max(e_rows(td.ns) - (td.ha - a), 0), e_rows(td.ns)) * td.ns + a0 - a * td.ns) * (RW * 64 / 16);
                }
                return RW == 16 ? (uint32_t)a0 * (RW * 64 / 16) : (uint32_t)min(max(4 - (td.ha - a0), 0), 4) * (RW * 64 / 16);
            };
            while (ok && next_unit()) {
                const int s_q[2] = {sq.pop(), sq.pop()};
                for (int c = td.c0; ok && c < td.nch; ++c) {
                    const int sk = sq.take();
                    sq.take();                       // (V)
                    if (c == td.c0) wait_full(s_q[0]);
                    wait_full(sk);
                    for (int hf = 0; hf < 2 && 4 * c + 2 * hf < td.ku; ++hf) {
                        const int left = td.ku - (4 * c + 2 * hf);
                        const uint32_t n = (left > 1 ? 8u : 4u) << 17, id = kIdS + n;
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            if (t >= td.ntq) break;
                            const unsigned buf = idx % NB;
                            if (t == 1 && c == td.c0 && hf == 0) wait_full(s_q[1]);
                            ok = ok && mbar_wait_all(bar(kBFree + buf), ((idx / NB) & 1) ^ 1u, cta_abort);
                            if (!ok) break;
                            ++idx;
                            tc_fence_after();
                            const uint32_t a = lo + s_q[t] * (L::kSlotB >> 4), b = lo + sk * (L::kSlotB >> 4) + hf * (64 * kRowB / 16), dst = tmem + 64u * buf;
                            const uint32_t ea = lo_e + mask_rows((td.tile0 + t) * kTileRows), eb = lo_e + mask_rows((2 * c + hf) * kG) + 2;
                            if (elect_one()) {
#pragma unroll
                                for (int ks = 0; ks < D / 16; ++ks) {
                                    const uint32_t oa = (ks / kPerPart) * (kTile * kRowB / 16) + (ks % kPerPart) * 2;
                                    if (ks == 0) mma_ss_h<false>(dst, a + oa, b + oa, hi, id);
                                    else mma_ss_h<true>(dst, a + oa, b + oa, hi, id);
                                }
                                if (td.flags & 4) mma_ss_h<true>(dst, ea, eb, hi_e, kIdE + n);
                                mma_commit(bar(kBS + buf));
                                if (c == td.nch - 1 && left <= 2) mma_commit(bar(kBEmpty + s_q[t]));
                                if (t == td.ntq - 1 && (hf == 1 || left <= 2)) mma_commit(bar(kBEmpty + sk));
                            }
                            __syncwarp();
                        }
                    }
                }
                sq.end_unit(s_q[0], s_q[1]);
            }
        } else if (warp == kPvWarp) {
            // -------------------------------------------------------------- O += P V
            constexpr uint32_t kIdO = make_idesc_elem(128, D, 0, 1);
            const uint64_t d_v = D == 32 ? make_sdesc_sw64_mn(smem0, 512, 512) : make_sdesc_sw128(smem0, kTile * kRowB);
            const uint32_t hi = sdesc_hi(d_v), lo = sdesc_lo(d_v);
            constexpr uint32_t kStep = 16 * kRowB / 16;
            SlotQueue<L::kSlots> sq;
            sq.init();
            uint32_t full_use = 0;
            unsigned idx = 0, opened[2] = {0, 0};
            bool ok = true;
            while (ok && next_unit()) {
                const int s_q[2] = {sq.pop(), sq.pop()};
                for (int c = td.c0; ok && c < td.nch; ++c) {
                    sq.take();                       // (K)
                    const int sv = sq.take();
                    ok = mbar_wait_all(bar(kBFullV + sv), (full_use >> sv) & 1, cta_abort);
                    full_use ^= 1u << sv;
                    for (int hf = 0; hf < 2 && 4 * c + 2 * hf < td.ku; ++hf) {
                        const int left = td.ku - (4 * c + 2 * hf);
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            if (t >= td.ntq) break;
                            const unsigned buf = idx % NB;
                            const bool first = c == td.c0 && hf == 0;
                            ok = ok && mbar_wait_all(bar(kBP + buf), (idx / NB) & 1, cta_abort);
                            if (first) {
                                ok = ok && mbar_wait_all(bar(kBOFree + t), (opened[t] & 1) ^ 1u, cta_abort);
                                ++opened[t];
                            }
                            if (!ok) break;
                            ++idx;
                            tc_fence_after();
                            const uint32_t dst = tmem + L::kColO + D * t, a = tmem + 64u * buf, b = lo + sv * (L::kSlotB >> 4) + hf * 4 * kStep;
                            if (elect_one()) {
                                if (first) mma_ts_h<false>(dst, a, b, hi, kIdO);
                                else mma_ts_h<true>(dst, a, b, hi, kIdO);
                                mma_ts_h<true>(dst, a + 8, b + kStep, hi, kIdO);
                                if (left > 1) {
                                    mma_ts_h<true>(dst, a + 16, b + 2 * kStep, hi, kIdO);
                                    mma_ts_h<true>(dst, a + 24, b + 3 * kStep, hi, kIdO);
                                }
                                mma_commit(bar(kBFree + buf));
                                if (c == td.nch - 1 && left <= 2) mma_commit(bar(kBO + t));
                                if (t == td.ntq - 1 && (hf == 1 || left <= 2)) mma_commit(bar(kBEmpty + sv));
                            }
                            __syncwarp();
                        }
                    }
                }
                sq.end_unit(s_q[0], s_q[1]);
            }
        }
    }

    // teardown: every role ends up here, also after an expired wait
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == kPvWarp) tmem_dealloc(tmem, 512);
    if (tid == 0 && *cta_abort) atomicExch(&g_fwd_win_timeout, 1);
}

// The bias tables of all heads as the softmax threads read them: bias log2 e by row and column difference, two copies.
template <int RW>
__global__ void swin_fwd_win_prep_kernel(const Geo g, const float* __restrict__ bias, float* __restrict__ tables) {
    let_dependents_start();
    const int per_head = Tab<RW>::rows(g.w) * Tab<RW>::kRowF, total = per_head * g.heads, nw = 2 * g.w - 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int head = i / per_head, e = i - head * per_head, row = e / Tab<RW>::kRowF, f = e - row * Tab<RW>::kRowF;
        const int c = f / Tab<RW>::kCopyF, da = row - Tab<RW>::kFront - (g.w - 1), db = f - c * Tab<RW>::kCopyF + c - (RW - 1);    // key minus query
        const bool in = da > -g.w && da < g.w && db > -g.w && db < g.w;
        tables[i] = in ? bias[((size_t)(g.w - 1 - da) * nw + (g.w - 1 - db)) * g.heads + head] * kLog2e : 0.f;
    }
}

// ST: by row difference, two copies (see Params).  Neighbouring threads read neighbouring heads and write a table each.
__global__ void swin_fwd_win_prep_strips_kernel(const Geo g, const float* __restrict__ bias, float* __restrict__ tables, int strips) {
    let_dependents_start();
    const int nw = 2 * g.w - 1, rl = 64 * strips, per_head = nw * 2 * rl;
    const long long total = (long long)per_head * g.heads;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int e = (int)(i / g.heads), head = (int)(i - (long long)e * g.heads);
        const int row = e / (2 * rl), f = e - row * 2 * rl, c = f / rl, db = f - c * rl + c - (32 * strips - 1);      // key minus query
        tables[(size_t)head * per_head + e] = db > -g.w && db < g.w ? __ldg(bias + ((size_t)(nw - 1 - row) * nw + (g.w - 1 - db)) * g.heads + head) * kLog2e : 0.f;
    }
}

}  // namespace

cudaError_t read_fwd_win_status(int* timed_out) {
    int zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(timed_out, g_fwd_win_timeout, sizeof(int));
    if (e != cudaSuccess) return e;
    if (*timed_out) e = cudaMemcpyToSymbol(g_fwd_win_timeout, &zero, sizeof(int));
    return e;
}

#ifndef TERRA_ELEM_F16
bool fwd_win_supported(const Geo& g) {
    // (head dim 32 with sides up to 16 has a kernel of its own, 0.77 against 1.16 ms on the 510 x 1080 grid with 12 heads)
    // The register-tile kernel packs a window's tokens densely; it is the faster one where a window fills little of the slots of this one.
    // Register tiles / this kernel, us, on 240 x 360, 2 x 121 x 250 and 96 x 180 tokens:
    //   head dim 32, side 17 214/495 400/1041 89/235, 22 302/340 556/709 123/159; 23 344/332 664/687 144/140, 24 326/258 611/638 136/126; sides
    //   above 24 work on all 32 slots of a row: 25 353/430 705/837 154/201, 26 392/402 736/830 164/169; 27 436/386 810/816 175/181, 28 463/342;
    //   head dim 64, side 9 226/318 212/349 52/80, 11 166/238 156/246 39/56; 12 267/183 248/214 60/46; 17 338/468 318/426 72/95; 18 416/358 379/368 95/84;
    //   head dim 128, this kernel at every side: 9 283/261 392/369 91/95, 10 242/238 338/328 74/82, 11 207/171 287/269 68/64, 17 400/346 558/486 123/118.
    // Strips: where the windows' work in them (strip_work) is at most 2.8 times the dense one at head dim 32, 6 times at 64 and 128, and the largest
    // window has more than 5, 4 and 2 blocks of 64 tokens (below, the two launches and a 128-slot tile's chain cost more than the register
    // tiles take in all).  Register tiles / strips, us, 6 x 32 channels: side 33 1020/1408 686/1019 216/306, 36 1183/1359 795/902 242/265, 38 1240/1388
    // 856/953 248/249, 40 1410/1304 966/1078 258/238, 44 1677/1394 1124/871 364/286; 6 x 64: side 33 1360/1260 916/931 287/296, 36 1584/1178 1066/849 324/247;
    // 4 x 128: side 33 1463/999 983/726 306/247.  Side 64 on narrow and low grids: 200 x 64 x 1, 6 x 32 23/3868; 200 x 8 x 8, 6 x 64 29/86.  On 1662
    // shapes of sides 33 .. 128 strips alone were more than 5 % slower on 574, by the rule the wrong one of the two is taken on 92.
    if (win_strips(g)) {
        const StripWork x = strip_work(g);
        const int blocks = (g.nmax + 63) / 64;
        if (g.d == 32 ? blocks <= 5 || 10 * x.strips > 28 * x.dense : blocks <= (g.d == 64 ? 4 : 2) || x.strips > 6 * x.dense) return false;
        return g.w <= kMaxWinW && (long long)g.B * g.H * g.W < 0x7fffffffLL && (long long)g.B * g.Mh * g.Mw * g.heads * 64 < 0x7fffffffLL;
    }
    const bool sparse = g.d == 32 ? g.w <= 22 || g.w == 25 || g.w == 26 : g.d == 64 && (g.w <= 11 || g.w == 17);
    return (g.d == 64 || g.d == 128 || (g.d == 32 && g.w > 16)) && !sparse && g.w > 8 && g.w <= kMaxOnePassW && (long long)g.B * g.H * g.W < 0x7fffffffLL &&
           (long long)g.B * g.Mh * g.Mw * g.heads * 4 < 0x7fffffffLL;
}

size_t fwd_win_workspace_bytes(const Geo& g) {
    if (win_strips(g)) return sizeof(float) * (size_t)g.heads * (2 * g.w - 1) * 128 * strips_of(g.w);
    return sizeof(float) * (size_t)g.heads * (win_row_slots(g) == 16 ? Tab<16>::rows(g.w) * Tab<16>::kRowF : Tab<32>::rows(g.w) * Tab<32>::kRowF);
}
#endif

namespace {
template <int D, int RW, int KC = 4, bool ST = false>
cudaError_t launch_win(const Geo& g, const void* q, const void* k, const void* v, const float* bias, void* o, float* lse, void* workspace,
                       int sm_count, cudaStream_t stream) {
    using L = Lay<D, RW, ST>;
    Params p;
    p.g = g;
    Maps<ST> mq, mk, mv;
    if (!make_win_cols(&p.cols, g) || !make_win_maps(&mq, p.cols, g, q, g.ts) || !make_win_maps(&mk, p.cols, g, k, g.ts) || !make_win_maps(&mv, p.cols, g, v, g.ts))
        return cudaErrorNotSupported;
    p.q = (const __nv_bfloat16*)q; p.k = (const __nv_bfloat16*)k; p.v = (const __nv_bfloat16*)v;
    p.tables = (const float*)workspace;
    p.strips = ST ? strips_of(g.w) : 1;
    const int row_slots = (ST ? strips_of(g.w < g.W ? g.w : g.W) : 1) * RW;
    auto tiles_of = [&](int rows) { return (rows * row_slots + kTile - 1) / kTile; };
    p.rows = g.H / g.w;
    auto plan = [&](int tiles) {
        p.tiles = tiles;
        p.units_win = (tiles_of(g.w) + tiles - 1) / tiles;
        p.units_row = (tiles_of(g.H - p.rows * g.w) + tiles - 1) / tiles;
        p.units = (long long)g.B * g.Mw * g.heads * ((long long)p.rows * p.units_win + (g.Mh - p.rows) * p.units_row);
    };
    p.part_ha = !g.ph && g.sh > 0 ? (g.H - g.sh) % g.w : 0;
    p.part_row = p.part_ha > 0 ? (g.H - g.sh) / g.w : -1;
    // One tile a unit has a unit's chain to itself: two thirds of a pair's time (32 x 64 tokens, 4 x 32, side 32: 27.7 -> 23.6 us a call).
    plan(1);
    if (p.units > sm_count) plan(2);
    // A CTA keeps to one head where that leaves no more than 1 SM in 20 idle: neighbouring CTAs then read the heads of the same
    // tokens at the same time.  Otherwise each CTA takes a run of the units in head-major order.
    const int bound = sm_count / g.heads * g.heads;
    p.head_slow = bound * 20 < sm_count * 19 && p.units > bound;
    const long long ctas = p.head_slow ? sm_count : bound > 0 ? bound : sm_count;
    const long long total = ST ? (long long)g.heads * (2 * g.w - 1) * 128 * p.strips : g.heads * Tab<RW>::rows(g.w) * Tab<RW>::kRowF;
    const unsigned pblocks = (unsigned)(total / 512 + 1 < 592 ? total / 512 + 1 : 592);
    prof_begin("swin_fwd_win_prep_kernel", stream);
    if (ST) swin_fwd_win_prep_strips_kernel<<<pblocks, 256, 0, stream>>>(g, bias, (float*)workspace, p.strips);
    else swin_fwd_win_prep_kernel<RW><<<pblocks, 256, 0, stream>>>(g, bias, (float*)workspace);
    count_launch(stream);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int part = p.part_row < 0 ? 0 : part_tiles(p.part_ha, g.H - p.part_row * g.w < g.w ? g.H - p.part_row * g.w : g.w, RW);
    const auto kernel = ST || (part > 0 && part % p.tiles == 0) ? swin_fwd_win_kernel<D, RW, KC, ST, true> : swin_fwd_win_kernel<D, RW, KC, ST, ST>;
    e = prepare_kernel((const void*)kernel, L::kSmemBytes);
    if (e != cudaSuccess) return e;
    prof_begin("swin_fwd_win_kernel", stream);
    e = launch_dependent(kernel, (unsigned)(p.units < ctas ? p.units : ctas), kThreads, L::kSmemBytes, stream, p, (__nv_bfloat16*)o, lse, mq, mk, mv);
    count_launch(stream);
    return e;
}
}  // namespace

cudaError_t launch_fwd_win(const Geo& g, const void* q, const void* k, const void* v, const float* bias, void* o, float* lse, void* workspace,
                           int sm_count, cudaStream_t stream) {
    if (win_strips(g)) {
        auto fn = g.d == 32 ? launch_win<32, 32, 4, true> : g.d == 64 ? launch_win<64, 32, 4, true> : launch_win<128, 32, 4, true>;
        return fn(g, q, k, v, bias, o, lse, workspace, sm_count, stream);
    }
    const bool wide = win_row_slots(g) == 32, narrow = g.w <= 24;
    switch (g.d) {
        case 32: return (narrow ? launch_win<32, 32, 3> : launch_win<32, 32>)(g, q, k, v, bias, o, lse, workspace, sm_count, stream);
        case 64: return (!wide ? launch_win<64, 16> : narrow ? launch_win<64, 32, 3> : launch_win<64, 32>)(g, q, k, v, bias, o, lse, workspace, sm_count, stream);
        default: return (!wide ? launch_win<128, 16> : narrow ? launch_win<128, 32, 3> : launch_win<128, 32>)(g, q, k, v, bias, o, lse, workspace, sm_count, stream);
    }
}

}  // namespace terra
