// ask_work.cuh -- device building blocks shared by the ASK launch chain
// (ask_kernels.cu: one level kernel per depth, then the leaf kernel) and the
// persistent batch kernel fed from a device work queue (ask_queue.cu):
// region records, the chunked perimeter query, and the leaf machinery (the
// coherent pre-pass over fresh pixels, the ring of survivors, the two-orbit
// refill round, parking and the batched finish of parked orbits).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ask_device.cuh"
#include "ask_internal.h"

namespace ask {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kNone = 0xffffffffu;

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(kFull, v, o);
    return v;
}


// ---------------------------------------------------------------------------
// Region records: uint2 for one frame, uint4 (with the frame id) for a batch.
// ---------------------------------------------------------------------------
template <bool BATCH>
struct Rec;
template <>
struct Rec<false> {
    using T = uint2;
    static __device__ __forceinline__ Region region(T e) { return unpack_region(e); }
    static __device__ __forceinline__ uint32_t frame(T) { return 0u; }
    static __device__ __forceinline__ T child(T, uint2 c) { return c; }
};
template <>
struct Rec<true> {
    using T = uint4;
    static __device__ __forceinline__ Region region(T e) { return unpack_region(make_uint2(e.x, e.y)); }
    static __device__ __forceinline__ uint32_t frame(T e) { return e.z; }
    static __device__ __forceinline__ T child(T p, uint2 c) { return make_uint4(c.x, c.y, p.z, 0u); }
};

// The parameters of the frame a region belongs to, at one level.
struct FView {
    uint32_t *map;
    PixelMap pm;
    uint32_t n, max_dwell, side, child_side, r;
    bool split;
};

__device__ __forceinline__ FView view_single(const LevelArgs &a)
{
    FView v;
    v.map = a.map;
    v.pm = a.pm;
    v.n = a.n;
    v.max_dwell = a.max_dwell;
    v.side = a.side;
    v.child_side = a.child_side;
    v.r = a.r;
    v.split = a.split != 0u;
    return v;
}

__device__ __forceinline__ FView view_frame(const FrameDesc *frames, uint32_t f, uint32_t level)
{
    const FrameDesc &d = frames[f];
    FView v;
    v.map = d.map;
    v.pm = d.pm;
    v.n = d.n;
    v.max_dwell = d.max_dwell;
    v.r = d.r;
    v.side = d.side[level];
    v.child_side = ceil_div_u32(v.side, v.r);
    v.split = level + 1u < d.levels;
    return v;
}

// Chunked queries of regions with longer perimeters skip the short first
// rounds of query_group: such regions are seldom uniform outside the set
// (without short rounds for any chunk level 2 at n = 16384, side 64, took 229
// us against 211, with them for every chunk level 0 the same as without).
constexpr uint32_t kShortRoundsMaxPerimeter = 512;

// Chunk c of the `chunks` of a large region's perimeter (P pixels), queried
// by one warp: the pixels c, c + chunks, c + 2 chunks, ..., so that every
// chunk, and every group of 32 * NS in it, is spread over the whole perimeter.  The
// region's state st: x = common dwell found so far (kNone: none yet), y = 1
// once two dwells are known to differ, z = chunks finished without.  Chunks
// of the same region run on other warps at the same time and stop as soon as
// one of them has set y.  Returns whether this chunk found the difference
// first (GROUP_DIFFER: the caller decides the region), found none
// (GROUP_SAME), or stopped because another did (GROUP_STOP).
template <int NS>
__device__ __forceinline__ uint32_t chunk_query(const FView &a, const Region &g, uint32_t P, uint32_t c,
                                                uint32_t chunks, uint4 *st, uint32_t lag,
                                                uint32_t lane, Updates &it)
{
    const volatile uint32_t *ps = reinterpret_cast<const volatile uint32_t *>(st);
    const uint32_t n = P > c ? (P - c + chunks - 1u) / chunks : 0u;
    const uint32_t rnd = P <= kShortRoundsMaxPerimeter ? 0u : 3u;
    constexpr uint32_t K = kQueryRound;
    for (uint32_t base = 0; base < n; base += 32u * NS) {
        uint32_t sx = 0, sy = 0, vmin = 0, vmax = 0;
        if (lane == 0) {
            sx = ps[0];
            sy = ps[1];
        }
        if (__shfl_sync(kFull, sy, 0))
            return GROUP_STOP;
        sx = __shfl_sync(kFull, sx, 0);
        const uint32_t r = spread_group<K, NS, true>(a.pm, a.max_dwell, g, c, chunks, base, P, rnd, sx, ps, lag,
                                               lane, vmin, vmax, it);
        if (r == GROUP_STOP)
            return r;
        bool differ = (r == GROUP_DIFFER);
        if (!differ) {
            uint32_t old = kNone;
            if (vmin == vmax && lane == 0)
                old = atomicCAS(&st->x, kNone, vmin);
            old = __shfl_sync(kFull, old, 0);
            differ = vmin != vmax || (old != kNone && old != vmin);
        }
        if (differ) {
            uint32_t first = 0;
            if (lane == 0)
                first = atomicExch(&st->y, 1u) == 0u ? 1u : 0u;
            return __shfl_sync(kFull, first, 0) ? GROUP_DIFFER : GROUP_STOP;
        }
    }
    return GROUP_SAME;
}

// After chunk_query: whether this warp decides the region, and how.  The warp
// that found the difference decides at once; with none, the warp that
// finishes the last of the chunks does (a chunk that found a difference never
// counts as finished, so exactly one warp decides).
__device__ __forceinline__ bool chunk_decides(uint32_t r, uint4 *st, uint32_t chunks, uint32_t lane,
                                              bool &uniform, uint32_t &wv)
{
    uniform = false;
    if (r != GROUP_SAME)
        return r == GROUP_DIFFER;
    uint32_t last = 0, x = 0;
    if (lane == 0) {
        __threadfence();
        last = (atomicAdd(&st->z, 1u) == chunks - 1u) ? 1u : 0u;
        if (last) {
            __threadfence();
            x = atomicAdd(&st->x, 0u);
        }
    }
    wv = __shfl_sync(kFull, x, 0);
    uniform = true;
    return __shfl_sync(kFull, last, 0) != 0u;
}

// ---------------------------------------------------------------------------
// Leaf machinery (see the leaf kernel in ask_kernels.cu)
// ---------------------------------------------------------------------------
constexpr int kRefillWarps = 8;    // warps per CTA
// Resident CTAs per SM that the registers have to allow: 3 leave 85 a thread, so
// nothing spills (5 CTAs, 48 registers and 60 bytes spilled took 1.08 ms at n =
// 16384, g=16 r=4 B=16, against 0.96).  A batch takes 72 and runs 3 CTAs; one
// frame takes 63 and runs 4.  Held to 3 its leaf kernel alone is faster, 0.933 ms
// against 0.956, but the chain is slower, probably because the CTAs that start
// while the level kernel before still holds a part of the SMs stay unevenly
// spread (n = 16384 1.62 -> 1.89 ms, n = 65536 9.90 -> 11.9, n = 3001 366 -> 397
// us).
constexpr int kRefillMinBlocks = 3;
constexpr int kSlots = 2;          // orbits per lane in the refill loop (four: 0.94-0.99 ms)
constexpr uint32_t kParkCap = 96;  // parked orbits per warp (fewer than 32 wait, a round adds 64)
constexpr uint32_t kRingCap = 96;  // survivors per warp (< 32 + 64: topped up while below 32)
constexpr uint32_t kRawCount = 0xffffffffu;  // count of an orbit that may not run in blocks
constexpr int kLeafUnroll = 32;    // updates per unchecked block of the refill loop (a power of
                                   // two), two blocks a round: with one block of 64 an orbit
                                   // that escapes is searched for 31 updates instead of 15
                                   // (64 frames in a batch: 38.8 ms against 38.0)
// Idle or waiting slots (of 64) before a warp parks and refills: that code
// costs about a third of a round, and most rounds end a few orbits.  At
// n = 16384 the leaf kernel took 1.097 ms with 1, 1.077 with 8, 1.095 with 16.
constexpr uint32_t kRefillSlots = 8;
constexpr int kPreBlock = 8;       // updates per unchecked block of the pre-pass (a power of two)
constexpr int kPrePass = 64;       // updates of the pre-pass (a multiple of kPreBlock)

// The output and pixel mapping of the frame a leaf belongs to.
struct LView {
    uint32_t *map;
    PixelMap pm;
    uint32_t n, max_dwell;
};

template <bool BATCH>
__device__ __forceinline__ LView leaf_view(const LeafArgs &a, uint32_t frame)
{
    LView v;
    if (BATCH) {
        const FrameDesc &d = a.frames[frame];
        v.map = d.map;
        v.pm = d.pm;
        v.n = d.n;
        v.max_dwell = d.max_dwell;
    } else {
        v.map = a.map;
        v.pm = a.pm;
        v.n = a.n;
        v.max_dwell = a.max_dwell;
    }
    return v;
}

template <bool BATCH>
__device__ __forceinline__ void store_dwell(const LeafArgs &a, uint32_t frame, uint32_t pix, uint32_t v)
{
    const LView f = leaf_view<BATCH>(a, frame);
    f.map[(size_t)(pix >> 16) * f.n + (pix & 0xffffu)] = v;
}

// Exact dwell of a parked orbit: s.xy = state after d updates, known to
// pass the test, s.zw = the state kLeafUnroll / 2 updates later (the block's
// midpoint), and "escaped, or d >= max_dwell" known to hold kLeafUnroll
// updates later.  Points where escape is not absorbing (count kRawCount, at
// z = 0) take the tested loop instead.  u = (count, py << 16 | px).
template <bool COUNT, bool BATCH>
__device__ __forceinline__ void finish_parked(const LeafArgs &a, float4 s, uint2 u, uint32_t frame,
                                              Updates &it)
{
    const LView v = leaf_view<BATCH>(a, frame);
    const uint32_t px = u.y & 0xffffu, py = u.y >> 16;
    const float2 c = pixel_c(v.pm, px, py);
    uint32_t d = u.x;
    float x = s.x, y = s.y;
    if (d == kRawCount) {
        d = 0;
        while (d < v.max_dwell && z_bounded(x, y)) {
            z_update(x, y, c.x, c.y);
            ++d;
        }
    } else if (d < v.max_dwell) {
        // invariant: count d passes (d < max_dwell) and the predicate holds
        // at d + 2h; halve h until the first count where it holds is d + 1.
        // The first halving uses the block's saved midpoint state.
        {
            const uint32_t h = (uint32_t)kLeafUnroll / 2u;
            const bool hit = (v.max_dwell - d <= h) || !z_bounded(s.z, s.w);
            if (!hit) {
                x = s.z;
                y = s.w;
                d += h;
            }
        }
#pragma unroll
        for (uint32_t h = (uint32_t)kLeafUnroll / 4u; h >= 1u; h >>= 1) {
            float tx = x, ty = y;
#pragma unroll
            for (uint32_t k = 0; k < h; ++k)
                z_update(tx, ty, c.x, c.y);
            const bool hit = (v.max_dwell - d <= h) || !z_bounded(tx, ty);
            if (!hit) {
                x = tx;
                y = ty;
                d += h;
            }
        }
        d += 1u;
    }
    v.map[(size_t)py * v.n + px] = d;
    if (COUNT)
        it += d;
}

// Deferred fills ride along the leaf pass.  The last warp of every CTA
// starts as a fill warp: it takes bands of the fill list (at most
// kFillBandPx pixels each, 128-bit stores) from a counter until none are
// left, then joins the leaf work; every warp that runs out of leaves helps
// with the bands still left.  The HBM writes so proceed beside the FP32 work
// of the other warps instead of in a kernel of their own (the bands and the
// leaves are disjoint pixels), and the fill code sits outside the refill
// loop, adding nothing to its registers.
template <bool BATCH>
__device__ __forceinline__ void drain_fills(const LeafArgs &a, uint32_t lane)
{
    const uint32_t nfill = min(a.ctr->fill_count, a.fill_cap);
    for (;;) {
        uint32_t fi = 0;
        if (lane == 0)
            fi = atomicAdd(&a.ctr->fill_work, 1u);
        fi = __shfl_sync(kFull, fi, 0);
        if (fi >= nfill)
            return;
        const uint4 e = a.fills[fi];
        const Region g = unpack_region(make_uint2(e.x, e.y));
        if (BATCH) {
            const FrameDesc &d = a.frames[e.w];
            fill_band_warp(d.map, d.n, g, e.z, lane);
        } else {
            fill_band_warp(a.map, a.n, g, e.z, lane);
        }
    }
}

// floor(q / w) for q < 2^22 given inv_w = 1/w rounded to float: (q + 1/2)/w
// lies at least 1/(2w) away from an integer, far more than the rounding of
// the two float operations, so truncation gives the exact quotient.
__device__ __forceinline__ uint32_t rows_in(uint32_t q, float inv_w)
{
    return __float2uint_rz(__fmul_rz(__uint2float_rn(q) + 0.5f, inv_w));
}


// One orbit slot of a lane in the refill loop.
struct Slot {
    float x, y, cr, ci;
    float bx, by;     // an earlier state of the orbit (see settle_slot)
    uint32_t d, pix;  // count (kRawCount: not to run in blocks), pixel (py << 16 | px)
    uint32_t frame;   // batch: the orbit's frame
    uint32_t lim;     // batch: slot_limit of its frame
    bool busy;
};

__device__ __forceinline__ void slot_reset(Slot &s)
{
    s.x = s.y = s.cr = s.ci = s.bx = s.by = 0.0f;
    s.d = s.pix = s.frame = s.lim = 0;
    s.busy = false;
}

// A whole unchecked block may run while d < limit: kLeafUnroll - 1 below
// max_dwell, 0 if no block fits.
__device__ __forceinline__ uint32_t block_limit(uint32_t max_dwell)
{
    return max_dwell >= (uint32_t)kLeafUnroll ? max_dwell - (uint32_t)kLeafUnroll + 1u : 0u;
}

template <bool BATCH>
__device__ __forceinline__ uint32_t slot_limit(const LeafArgs &a, const Slot &s)
{
    return BATCH ? s.lim : block_limit(a.max_dwell);
}

// The warp's current leaf, handed out as a row-major cursor.  It lives in
// shared memory between pre-passes, out of the refill loop's registers.
struct LeafCursor {
    uint32_t rem, row0, col0, ox, oy, cw, frame;
    float inv_cw;
};

// An empty cursor (lane 0 writes, the warp sees it).
__device__ __forceinline__ void cursor_reset(LeafCursor &lc, uint32_t lane)
{
    if (lane == 0) {
        lc.rem = lc.row0 = lc.col0 = lc.ox = lc.oy = lc.frame = 0;
        lc.cw = 1;
        lc.inv_cw = 1.0f;
    }
    __syncwarp();
}

// A warp's share of the leaf kernel's shared memory: parked orbits (the
// states at their block's start and midpoint; count and pixel), the ring of
// survivors (state, pixel, count) and the leaf cursor.
template <bool BATCH>
struct WarpLeaf {
    float4 park_s[kParkCap];
    float4 ring[kRingCap];
    uint2 park_u[kParkCap];
    uint32_t park_f[BATCH ? kParkCap : 1], ring_f[BATCH ? kRingCap : 1];  // frames
    LeafCursor cursor;
};

// Warp-uniform fill levels: parked orbits, the ring's first entry and entries.
struct WarpFill {
    uint32_t parked, ring_h, ring_n;
};

__device__ __forceinline__ unsigned lanes_below()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Where the pre-pass takes its leaves from.
enum : uint32_t {
    SRC_MORE = 0,  // a leaf was given, or more may be asked for
    SRC_WAIT = 1,  // none is ready now, more may come (persistent batch kernel)
    SRC_DONE = 2,  // the leaves have run out
};

// Point the cursor at leaf region g of `frame`: its interior only when the
// perimeters are already in the map (a leaf of side <= 2 is all perimeter).
__device__ __forceinline__ void cursor_at(LeafCursor &lc, const Region &g, uint32_t frame,
                                          bool skip_perimeter)
{
    lc.frame = frame;
    if (skip_perimeter) {
        lc.cw = g.w > 2u ? g.w - 2u : 1u;
        lc.rem = (g.w > 2u && g.h > 2u) ? (g.w - 2u) * (g.h - 2u) : 0u;
        lc.ox = g.x0 + 1u;
        lc.oy = g.y0 + 1u;
    } else {
        lc.cw = g.w;
        lc.rem = g.w * g.h;
        lc.ox = g.x0;
        lc.oy = g.y0;
    }
    lc.row0 = lc.col0 = 0;
    lc.inv_cw = 1.0f / (float)lc.cw;
}

// Region tables and leaf lists are filled from both ends: `front` entries
// from slot 0 up (the regions or leaves likely to hold long orbits, or every
// entry where the producer does not order them) and the rest from slot
// cap - 1 down.  Entry t of the order in which they are taken (the front
// first, then the back in append order) sits at this slot.
__device__ __forceinline__ uint32_t table_slot(uint32_t t, uint32_t front, uint32_t cap)
{
    return t < front ? t : cap - 1u - (t - front);
}

// Entries of the front and of the whole list, within `cap`.  More leaves
// than `cap` (front and back met) latch the overflow error; block 0 reports.
__device__ __forceinline__ void leaf_extent(DevCounters *ctr, uint32_t cap, uint32_t &front,
                                            uint32_t &total)
{
    const uint32_t h = ctr->leaf_count, l = ctr->leaf_light;
    front = min(h, cap);
    total = front + min(l, cap - front);
    if (blockIdx.x == 0 && threadIdx.x == 0 && (unsigned long long)h + l > cap)
        atomicOr(&ctr->error, ERR_LEAF_OVERFLOW);
}

// The leaf list of a launch chain: complete when the leaf kernel starts, its
// leaves (or row bands of them, see leaf_item_shift) handed out one at a time
// by a device counter.
template <bool BATCH>
struct LeafList {
    const typename Rec<BATCH>::T *leaves;
    uint32_t cap;
    const uint3 *extent;  // in shared memory: entries of the front, entries,
                          // shift (an item is one of 1 << shift bands of a leaf)

    __device__ __forceinline__ uint32_t next(const LeafArgs &a, LeafCursor &lc, uint32_t lane)
    {
        using R = Rec<BATCH>;
        uint32_t li = 0;
        if (lane == 0)
            li = atomicAdd(&a.ctr->leaf_work, 1u);
        li = __shfl_sync(kFull, li, 0);
        const uint32_t shift = extent->z, leaf = li >> shift;
        if (leaf >= extent->y)
            return SRC_DONE;
        const typename R::T e = leaves[table_slot(leaf, extent->x, cap)];
        const Region g = R::region(e);
        const bool skip = a.skip_perimeter != 0u;
        if (shift) {
            // rows [r0, r1) of the rows to compute (a leaf of fewer rows than
            // bands has empty ones)
            const uint32_t band = li & ((1u << shift) - 1u);
            const bool inner = skip && g.w > 2u && g.h > 2u;
            const uint32_t rows = inner ? g.h - 2u : g.h;
            const uint32_t r0 = (uint32_t)(((unsigned long long)rows * band) >> shift);
            const uint32_t r1 = (uint32_t)(((unsigned long long)rows * (band + 1u)) >> shift);
            if (r0 == r1 || (skip && !inner)) {
                lc.rem = 0;
                return SRC_MORE;
            }
            cursor_at(lc, g, R::frame(e), skip);
            lc.oy += r0;
            lc.rem = (r1 - r0) * lc.cw;
            return SRC_MORE;
        }
        cursor_at(lc, g, R::frame(e), skip);
        return SRC_MORE;
    }
};

// Put a survivor on the ring, `rank` entries past its end.
template <bool BATCH>
__device__ __forceinline__ void push_survivor(WarpLeaf<BATCH> &w, const WarpFill &f, uint32_t rank,
                                              float x, float y, uint32_t pix, uint32_t d, uint32_t frame)
{
    uint32_t k = f.ring_h + f.ring_n + rank;
    if (k >= kRingCap)
        k -= kRingCap;
    w.ring[k] = make_float4(x, y, __uint_as_float(pix), __uint_as_float(d));
    if (BATCH)
        w.ring_f[k] = frame;
}

// Pre-pass: up to 64 fresh pixels from the leaf cursor, the j-th on lane
// j & 31 (two a lane, side by side), run their first kPrePass updates in
// lockstep: unchecked blocks of kPreBlock, one test each, only while a whole
// block stays within max_dwell.  A pixel whose block fails the test goes back
// to the block's start and repeats it (with the same end) until every pixel
// has failed or the pass is over.  A failed block holds the pixel's dwell: a
// binary search over it (kPreBlock - 1 updates and log2(kPreBlock) tests, the
// same on every lane) finds it, and the dwell is written.  Every other pixel
// is pushed onto the ring with its state: survivors of the whole pass, orbits
// stopped by max_dwell, and points where escape is not absorbing (kRawCount;
// the refill loop parks them and finish_parked runs the tested loop).  Leaves
// come from `src` (see LeafList); `srcst` becomes SRC_WAIT or SRC_DONE when it
// has none to give.  Returns the number of pixels taken.
template <bool COUNT, bool BATCH, typename Src>
__device__ __forceinline__ uint32_t pre_pass(const LeafArgs &a, Src &src, uint32_t &srcst,
                                             WarpLeaf<BATCH> &w, WarpFill &f, uint32_t lane,
                                             Updates &it, unsigned long long &lpx)
{
    uint32_t pix0 = 0, pix1 = 0, fr0 = 0, fr1 = 0;
    uint32_t base = 0;
    LeafCursor lc = w.cursor;
    while (base < 64u && srcst == SRC_MORE) {
        if (lc.rem == 0) {
            srcst = src.next(a, lc, lane);
            continue;
        }
        const uint32_t take = min(64u - base, lc.rem);
        const uint32_t j0 = lane - base, j1 = lane + 32u - base;  // (wrap below base)
        if (j0 < take) {
            const uint32_t q = lc.col0 + j0, dr = rows_in(q, lc.inv_cw);
            pix0 = ((lc.oy + lc.row0 + dr) << 16) | (lc.ox + q - dr * lc.cw);
            fr0 = lc.frame;
        }
        if (j1 < take) {
            const uint32_t q = lc.col0 + j1, dr = rows_in(q, lc.inv_cw);
            pix1 = ((lc.oy + lc.row0 + dr) << 16) | (lc.ox + q - dr * lc.cw);
            fr1 = lc.frame;
        }
        const uint32_t q = lc.col0 + take, dr = rows_in(q, lc.inv_cw);
        lc.col0 = q - dr * lc.cw;
        lc.row0 += dr;
        lc.rem -= take;
        base += take;
    }
    __syncwarp();
    if (lane == 0)
        w.cursor = lc;
    __syncwarp();
    if (base == 0)
        return 0;
    const bool have0 = lane < base, have1 = lane + 32u < base;
    const float2 c0 = pixel_c(leaf_view<BATCH>(a, fr0).pm, pix0 & 0xffffu, pix0 >> 16);
    const float2 c1 = pixel_c(leaf_view<BATCH>(a, fr1).pm, pix1 & 0xffffu, pix1 >> 16);
    const uint32_t cap0 = leaf_view<BATCH>(a, fr0).max_dwell, cap1 = leaf_view<BATCH>(a, fr1).max_dwell;
    const bool go0 = have0 && escape_absorbing(c0.x, c0.y);
    const bool go1 = have1 && escape_absorbing(c1.x, c1.y);
    const f32x2 cr = pack2(c0.x, c1.x), ci = pack2(c0.y, c1.y);
    constexpr uint32_t KP = (uint32_t)kPreBlock;
    float x0 = 0.0f, y0 = 0.0f, x1 = 0.0f, y1 = 0.0f;
    uint32_t d0 = 0, d1 = 0;
    bool run0 = go0, run1 = go1;  // passed every block so far
    // one frame: the blocks that fit below max_dwell, the same for every lane
    const uint32_t nb = BATCH ? (uint32_t)(kPrePass / kPreBlock)
                              : min((uint32_t)(kPrePass / kPreBlock), a.max_dwell / KP);
#pragma unroll
    for (int b = 0; b < kPrePass / kPreBlock; ++b) {
        if (!BATCH && (uint32_t)b >= nb)
            break;
        f32x2 x = pack2(x0, x1), y = pack2(y0, y1);
#pragma unroll
        for (int k = 0; k < kPreBlock; ++k)
            z_update2(x, y, cr, ci);
        float m0, m1, e0, e1;
        unpack2(fma2(x, x, mul2(y, y)), m0, m1);
        run0 = go0 && m0 < 4.0f && (!BATCH || cap0 - d0 >= KP);
        run1 = go1 && m1 < 4.0f && (!BATCH || cap1 - d1 >= KP);
        unpack2(x, e0, e1);
        x0 = run0 ? e0 : x0;
        x1 = run1 ? e1 : x1;
        unpack2(y, e0, e1);
        y0 = run0 ? e0 : y0;
        y1 = run1 ? e1 : y1;
        d0 += run0 ? KP : 0u;
        d1 += run1 ? KP : 0u;
        if (!__any_sync(kFull, run0 || run1))
            break;
    }
    const bool esc0 = go0 && !run0 && (!BATCH || cap0 - d0 >= KP);
    const bool esc1 = go1 && !run1 && (!BATCH || cap1 - d1 >= KP);
    if (__any_sync(kFull, esc0 || esc1)) {
        // invariant: the state at count r passes the test and the state at
        // r + 2h fails; halve h until the first failing count is r + 1
        float rx0 = x0, ry0 = y0, rx1 = x1, ry1 = y1;
        uint32_t r0 = d0, r1 = d1;
#pragma unroll
        for (uint32_t h = KP / 2u; h >= 1u; h >>= 1) {
            f32x2 x = pack2(rx0, rx1), y = pack2(ry0, ry1);
#pragma unroll
            for (uint32_t k = 0; k < h; ++k)
                z_update2(x, y, cr, ci);
            float m0, m1, e0, e1;
            unpack2(fma2(x, x, mul2(y, y)), m0, m1);
            unpack2(x, e0, e1);
            rx0 = m0 < 4.0f ? e0 : rx0;
            rx1 = m1 < 4.0f ? e1 : rx1;
            unpack2(y, e0, e1);
            ry0 = m0 < 4.0f ? e0 : ry0;
            ry1 = m1 < 4.0f ? e1 : ry1;
            r0 += m0 < 4.0f ? h : 0u;
            r1 += m1 < 4.0f ? h : 0u;
        }
        if (esc0) {
            store_dwell<BATCH>(a, fr0, pix0, r0 + 1u);
            if (COUNT) {
                it += r0 + 1u;
                ++lpx;
            }
        }
        if (esc1) {
            store_dwell<BATCH>(a, fr1, pix1, r1 + 1u);
            if (COUNT) {
                it += r1 + 1u;
                ++lpx;
            }
        }
    }
    const bool push0 = have0 && !esc0, push1 = have1 && !esc1;
    const unsigned p0 = __ballot_sync(kFull, push0), p1 = __ballot_sync(kFull, push1);
    const unsigned lt = lanes_below();
    if (push0)
        push_survivor<BATCH>(w, f, (uint32_t)__popc(p0 & lt), x0, y0, pix0, go0 ? d0 : kRawCount, fr0);
    if (push1)
        push_survivor<BATCH>(w, f, (uint32_t)(__popc(p0) + __popc(p1 & lt)), x1, y1, pix1,
                             go1 ? d1 : kRawCount, fr1);
    f.ring_n += (uint32_t)(__popc(p0) + __popc(p1));
    __syncwarp();
    return base;
}

// Take ring entry `rank` from the front into an idle slot.
template <bool BATCH>
__device__ __forceinline__ void take_survivor(const LeafArgs &a, const WarpLeaf<BATCH> &w,
                                              const WarpFill &f, uint32_t rank, Slot &s)
{
    uint32_t k = f.ring_h + rank;
    if (k >= kRingCap)
        k -= kRingCap;
    const float4 e = w.ring[k];
    s.frame = BATCH ? w.ring_f[k] : 0u;
    s.pix = __float_as_uint(e.z);
    s.d = __float_as_uint(e.w);
    const LView v = leaf_view<BATCH>(a, s.frame);
    const float2 c = pixel_c(v.pm, s.pix & 0xffffu, s.pix >> 16);
    s.x = s.bx = e.x;
    s.y = s.by = e.y;
    s.cr = c.x;
    s.ci = c.y;
    if (BATCH)
        s.lim = block_limit(v.max_dwell);
    s.busy = true;
}

// Refill the idle slots of the refill loop from the ring of survivors: slot 0
// of the idle lanes first, then slot 1, ...  Returns the orbits taken.
template <bool BATCH, int NS>
__device__ __forceinline__ uint32_t refill_from_ring(const LeafArgs &a, const WarpLeaf<BATCH> &w,
                                                     WarpFill &f, Slot *s)
{
    const unsigned lt = lanes_below();
    uint32_t n = 0;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const unsigned idle = __ballot_sync(kFull, !s[i].busy);
        const uint32_t r = n + (uint32_t)__popc(idle & lt);
        if (!s[i].busy && r < f.ring_n)
            take_survivor<BATCH>(a, w, f, r, s[i]);
        n += (uint32_t)__popc(idle);
    }
    n = min(n, f.ring_n);
    f.ring_h += n;
    if (f.ring_h >= kRingCap)
        f.ring_h -= kRingCap;
    f.ring_n -= n;
    __syncwarp();
    return n;
}

// Orbits in the first NS slots of the warp.
template <int NS>
__device__ __forceinline__ uint32_t busy_slots(const Slot *s)
{
    uint32_t n = 0;
#pragma unroll
    for (int i = 0; i < NS; ++i)
        n += (uint32_t)__popc(__ballot_sync(kFull, s[i].busy));
    return n;
}

// Move the orbits of slot 1 onto the ring (the ring and both slots hold at
// most 32 orbits between them when this is called), so the refill that
// follows puts every orbit in slot 0 and the rounds after it update one
// orbit per lane: once the leaves have run out and few orbits are left, a
// round then costs half the work.
template <bool BATCH>
__device__ __forceinline__ void fold_slot1(WarpLeaf<BATCH> &w, WarpFill &f, Slot &s1)
{
    const unsigned b = __ballot_sync(kFull, s1.busy);
    if (s1.busy) {
        push_survivor<BATCH>(w, f, (uint32_t)__popc(b & lanes_below()), s1.x, s1.y, s1.pix, s1.d, s1.frame);
        s1.busy = false;
    }
    f.ring_n += (uint32_t)__popc(b);
    __syncwarp();
}

// Settle a slot after a round's second block (x, y: the state after it): an
// orbit that passed the block's test counts it, and is done, at max_dwell, when
// it has got there (the block limit lim stands kLeafUnroll - 1 below max_dwell)
// or when its state equals the saved one (bx, by): the iteration is a function of the
// state alone, so an orbit that repeats a state repeats it for ever and never
// escapes.  (Equal up to the sign of a zero, which changes no magnitude and
// no test.)  The saved state is renewed whenever d / K is a power of two, so a
// cycle is seen within twice the updates it took to enter it, if its length
// divides a multiple of K below d.  An orbit that failed the test, or has less
// than a block left, stays at the block's start and waits there to be parked
// (running the block again changes nothing).  Returns whether it waits.
template <bool COUNT, bool BATCH>
__device__ __forceinline__ bool settle_slot(const LeafArgs &a, Slot &s, float x, float y,
                                            Updates &it, unsigned long long &lpx)
{
    const uint32_t K = 2u * (uint32_t)kLeafUnroll;
    const uint32_t lim = slot_limit<BATCH>(a, s);
    const bool ok = s.d < lim && z_bounded(x, y);
    if (ok) {
        s.x = x;
        s.y = y;
        s.d += (uint32_t)kLeafUnroll;
    }
    const uint32_t md = lim + (uint32_t)kLeafUnroll - 1u;
    const bool end = s.busy && lim != 0u && s.d == md;
    if (end || (s.busy && ok && x == s.bx && y == s.by)) {
        store_dwell<BATCH>(a, s.frame, s.pix, md);
        if (COUNT) {
            it += md;
            it.spared += md - s.d;
            ++lpx;
        }
        s.busy = false;
    } else if (ok && ((s.d / K) & (s.d / K - 1u)) == 0u) {
        s.bx = x;
        s.by = y;
    }
    return s.busy && !ok;
}

// kLeafUnroll / 2 unchecked updates of one or two orbits.
template <int NS>
__device__ __forceinline__ void half_block(float *x, float *y, const float *cr, const float *ci)
{
    if (NS == 1) {
#pragma unroll
        for (int k = 0; k < kLeafUnroll / 2; ++k)
            z_update(x[0], y[0], cr[0], ci[0]);
    } else {
        f32x2 X = pack2(x[0], x[NS - 1]), Y = pack2(y[0], y[NS - 1]);
        const f32x2 CR = pack2(cr[0], cr[NS - 1]), CI = pack2(ci[0], ci[NS - 1]);
#pragma unroll
        for (int k = 0; k < kLeafUnroll / 2; ++k)
            z_update2(X, Y, CR, CI);
        unpack2(X, x[0], x[NS - 1]);
        unpack2(Y, y[0], y[NS - 1]);
    }
}

// One round of the refill loop: two unchecked blocks of kLeafUnroll updates on
// the first NS slots (the results of an idle slot are not used; an orbit that
// fails the first block repeats it as its second), and what follows for each
// slot (settle_slot).  Once `thr` slots or more are idle or
// wait, the waiting orbits are parked (the state before the block and the
// block's midpoint state go to the park buffer), and whenever 32 orbits are
// parked the warp finishes them together.  Returns whether `thr` was reached.
template <bool COUNT, bool BATCH, int NS>
__device__ __forceinline__ bool refill_round(const LeafArgs &a, WarpLeaf<BATCH> &w, WarpFill &f,
                                             Slot *s, uint32_t thr, uint32_t lane,
                                             Updates &it, unsigned long long &lpx)
{
    float x[NS], y[NS], cr[NS], ci[NS], mx[NS], my[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        x[i] = s[i].x;
        y[i] = s[i].y;
        cr[i] = s[i].cr;
        ci[i] = s[i].ci;
    }
    // first block: an orbit that passes it moves on, another repeats it below
    half_block<NS>(x, y, cr, ci);
    half_block<NS>(x, y, cr, ci);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        if (s[i].d < slot_limit<BATCH>(a, s[i]) && z_bounded(x[i], y[i])) {
            s[i].x = x[i];
            s[i].y = y[i];
            s[i].d += (uint32_t)kLeafUnroll;
        } else {
            x[i] = s[i].x;
            y[i] = s[i].y;
        }
    }
    half_block<NS>(x, y, cr, ci);
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        mx[i] = x[i];
        my[i] = y[i];
    }
    half_block<NS>(x, y, cr, ci);
    bool wait[NS];
    uint32_t still = 0;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        wait[i] = settle_slot<COUNT, BATCH>(a, s[i], x[i], y[i], it, lpx);
        still += (uint32_t)__popc(__ballot_sync(kFull, wait[i] || !s[i].busy));
    }
    if (still < thr)
        return false;
    const unsigned lt = lanes_below();
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const unsigned p = __ballot_sync(kFull, wait[i]);
        if (wait[i]) {
            const uint32_t k = f.parked + (uint32_t)__popc(p & lt);
            w.park_s[k] = make_float4(s[i].x, s[i].y, mx[i], my[i]);
            w.park_u[k] = make_uint2(s[i].d, s[i].pix);
            if (BATCH)
                w.park_f[k] = s[i].frame;
            s[i].busy = false;
        }
        f.parked += (uint32_t)__popc(p);
    }
    __syncwarp();
    while (f.parked >= 32u) {
        f.parked -= 32u;
        const uint32_t k = f.parked + lane;
        const float4 sv = w.park_s[k];
        const uint2 uv = w.park_u[k];
        const uint32_t fr = BATCH ? w.park_f[k] : 0u;
        __syncwarp();
        finish_parked<COUNT, BATCH>(a, sv, uv, fr, it);
        if (COUNT)
            ++lpx;
    }
    return true;
}

// Move the ring's survivors to the pool; false once the pool is full (what did
// not fit stays on the ring).
template <bool BATCH>
__device__ __forceinline__ bool pool_survivors(const LeafArgs &a, const WarpLeaf<BATCH> &w, WarpFill &f,
                                               uint32_t lane)
{
    uint32_t base = 0;
    if (lane == 0 && f.ring_n)
        base = atomicAdd(&a.ctr->pool_count, f.ring_n);
    base = __shfl_sync(kFull, base, 0);
    const uint32_t fit = base < a.pool_cap ? min(f.ring_n, a.pool_cap - base) : 0u;
    for (uint32_t k = lane; k < fit; k += 32u) {
        uint32_t j = f.ring_h + k;
        if (j >= kRingCap)
            j -= kRingCap;
        a.pool[base + k] = w.ring[j];
        if (BATCH)
            a.pool_frame[base + k] = w.ring_f[j];
    }
    f.ring_h += fit;
    if (f.ring_h >= kRingCap)
        f.ring_h -= kRingCap;
    f.ring_n -= fit;
    __syncwarp();
    return f.ring_n == 0u;
}

// Survivors from the pool, kPoolTake at a time onto the ring: a warp's first
// ones by its number, the others by a counter.
constexpr uint32_t kPoolTake = 32;
struct PoolFeed {
    uint32_t total, next, first_end;  // entries; the warp's next; where the counter's begin

    __device__ __forceinline__ void operator()(const LeafArgs &a, uint32_t &srcst, WarpLeaf<true> &w,
                                               WarpFill &f, uint32_t lane, Updates &,
                                               unsigned long long &)
    {
        if (next == kNone) {
            if (lane == 0)
                next = first_end + atomicAdd(&a.ctr->pool_work, kPoolTake);
            next = __shfl_sync(kFull, next, 0);
        }
        if (next >= total) {
            srcst = SRC_DONE;
            return;
        }
        const uint32_t n = min(kPoolTake, total - next);
        if (lane < n) {
            const float4 e = a.pool[next + lane];
            push_survivor<true>(w, f, lane, e.x, e.y, __float_as_uint(e.z), __float_as_uint(e.w),
                                a.pool_frame[next + lane]);
        }
        f.ring_n += n;
        next = kNone;
        __syncwarp();
    }
};

// Survivors of pre-passes over the pixels of a source.
template <bool COUNT, bool BATCH, typename Src>
struct PrePassFeed {
    Src &src;

    __device__ __forceinline__ void operator()(const LeafArgs &a, uint32_t &srcst, WarpLeaf<BATCH> &w,
                                               WarpFill &f, uint32_t lane, Updates &it,
                                               unsigned long long &lpx)
    {
        pre_pass<COUNT, BATCH>(a, src, srcst, w, f, lane, it, lpx);
    }
};

// Refill rounds over the survivors that `feed` puts on the ring, until it has
// run out (srcst) and no orbit is left but the fewer than 32 still parked.
template <bool COUNT, bool BATCH, typename Feed>
__device__ __forceinline__ void run_orbits(const LeafArgs &a, Feed &feed, uint32_t srcst,
                                           WarpLeaf<BATCH> &w, WarpFill &f, uint32_t lane,
                                           Updates &it, unsigned long long &lpx)
{
    Slot s[kSlots];
#pragma unroll
    for (int i = 0; i < kSlots; ++i)
        slot_reset(s[i]);
    for (;;) {
        // refill idle slots from the ring, topping it up while it holds fewer
        // survivors than idle slots (at most 32)
        for (;;) {
            const uint32_t idle = 32u * kSlots - busy_slots<kSlots>(s);
            if (idle < kRefillSlots || (srcst != SRC_MORE && f.ring_n == 0))
                break;
            const uint32_t want = min(idle, 32u);
            while (f.ring_n < want && srcst == SRC_MORE)
                feed(a, srcst, w, f, lane, it, lpx);
            refill_from_ring<BATCH, kSlots>(a, w, f, s);
        }
        // once the source has run out and the orbits left fit in one slot
        // per lane, the tail runs on slot 0 alone
        if (srcst != SRC_MORE && f.ring_n + busy_slots<kSlots>(s) <= 32u)
            break;
        while (!refill_round<COUNT, BATCH, kSlots>(a, w, f, s, kRefillSlots, lane, it, lpx)) {
        }
    }
    fold_slot1<BATCH>(w, f, s[1]);
    refill_from_ring<BATCH, 1>(a, w, f, s);
    while (!refill_round<COUNT, BATCH, 1>(a, w, f, s, 32u, lane, it, lpx)) {
    }
}

// The orbits still parked after run_orbits, and the warp's counts.
template <bool COUNT, bool BATCH>
__device__ __forceinline__ void finish_orbits(const LeafArgs &a, const WarpLeaf<BATCH> &w, const WarpFill &f,
                                              uint32_t lane, Updates it, unsigned long long lpx)
{
    if (lane < f.parked) {
        finish_parked<COUNT, BATCH>(a, w.park_s[lane], w.park_u[lane], BATCH ? w.park_f[lane] : 0u, it);
        if (COUNT)
            ++lpx;
    }
    if (COUNT) {
        count_updates(a.ctr, &a.ctr->leaf_iters, &a.ctr->leaf_spared, it, lane);
        lpx = warp_sum_u64(lpx);
        if (lane == 0 && lpx)
            atomicAdd(&a.ctr->leaf_pixels, lpx);
    }
}

}  // namespace ask
