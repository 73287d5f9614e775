// ask_kernels.cu -- exhaustive kernel and the Adaptive Serial Kernels (ASK)
// pipeline: init, one level kernel per subdivision depth, leaf kernel (which
// also writes the deferred fills), and the fill kernel of the variants that
// fill in a pass of their own.
//
// ASK (paper Sec. 5): the active regions of depth i sit in a device-resident
// offset lookup table (read-OLT, Sec. 5.2).  One kernel per depth evaluates
// every region's perimeter (the exploration query Q of Sec. 4.2.1), fills
// uniform regions (terminal work T), and appends the r x r sub-regions of the
// others to the write-OLT with atomic adds on a global counter (Sec. 5.3.1);
// the counter's final value is the next depth's region count.  The tables are
// swapped between depths (Sec. 5.3.2).  Regions that may not split further
// go to a leaf list, evaluated pixel by pixel by the last kernel (the final
// terminal pass of Sec. 5.1, L(n, tau) of Sec. 4.2).
//
// GB300 layout of that scheme:
//  * level kernels are persistent (a grid sized to the SM count), read the
//    region count from device memory and hand out work with an atomic
//    counter, so no depth needs a host round trip;
//  * a work item is one region's perimeter, or one chunk of kChunkPx
//    perimeter pixels of a large region (a batch: see plan_batch; several
//    warps per region: the MBR mapping of Sec. 4.3.2 applied to the query), one
//    warp per item;
//  * each region table is filled from both ends (regions whose centre orbit
//    stays bounded for a short probe from the front), so a level kernel
//    takes its longest regions first; the leaf list likewise;
//  * a query stops at the first two perimeter dwells known to differ; warps
//    of one region share that verdict through a per-region state word; the
//    warp that finds the difference, or finishes the region's last chunk
//    without one, takes the decision;
//  * orbits proven to stay in the set (capture_disc, repeated states) end
//    there, with the dwell they would have had;
//  * decisions are compacted per warp: each lane keeps the outcome of one
//    region, then one atomicAdd per list serves up to 32 regions (the
//    block-scan + single atomic alternative of Sec. 5.3.1, at warp scope);
//  * small uniform regions are filled in place by their warp; large ones go
//    to a fill list as bands of rows, written with 128-bit stores by the
//    leaf kernel's fill warps beside its FP32 work (or by the fill kernel);
//  * the OLTs are preallocated for the worst case, so nothing is resized
//    between depths (Sec. 5.3.2 reallocates instead).
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "ask_device.cuh"
#include "ask_internal.h"
#include "ask_launch.cuh"
#include "ask_work.cuh"

namespace ask {

namespace {

constexpr uint32_t kWarpStage = 512;  // staged perimeter pixels per warp (exact last level)
constexpr int kOrderProbe = 64;       // updates of the order probe (region_probe)

enum : uint32_t { KIND_NONE = 0, KIND_FILL = 1, KIND_SPLIT = 2, KIND_LEAF = 3, KIND_FILL_LATER = 4 };

// ---------------------------------------------------------------------------
// Exhaustive: one thread per pixel over a flat grid of block_x x block_y
// tiles (paper Sec. 4.1: |G_E| = n^2 threads, work n^2 A).
// ---------------------------------------------------------------------------
template <bool COUNT>
__global__ void __launch_bounds__(1024) exhaustive_kernel(uint32_t *__restrict__ map, uint32_t n,
                                                          PixelMap pm, uint32_t max_dwell,
                                                          uint32_t tiles_x, DevCounters *ctr)
{
    const uint32_t tile = blockIdx.x;
    const uint32_t ty = tile / tiles_x, tx = tile - ty * tiles_x;
    const uint32_t px = tx * blockDim.x + threadIdx.x;
    const uint32_t py = ty * blockDim.y + threadIdx.y;
    Updates it;
    if (px < n && py < n) {
        const float2 c = pixel_c(pm, px, py);
        const uint32_t d = dwell(c.x, c.y, max_dwell, COUNT ? &it.spared : nullptr);
        map[(size_t)py * n + px] = d;
        it += d;
    }
    if (COUNT)
        count_updates(ctr, nullptr, nullptr, it, (threadIdx.x + threadIdx.y * blockDim.x) % 32u);
}

// Order probe of a region (the order in which the region tables and the
// leaf list are taken): does the orbit of the region's centre pixel stay
// bounded for kOrderProbe updates?  Regions inside the set, whose perimeter
// orbits all run to max_dwell, and leaves holding such orbits answer yes;
// taking them first lets a kernel's warps run out of work together instead
// of ending on a wave of its longest items.  Only the order of the work
// depends on it, never a dwell.  Unchecked updates: an escaped orbit runs to
// inf or NaN and fails the test; where escape is not absorbing the answer is
// no.
__device__ __forceinline__ bool region_probe(const PixelMap &pm, const Region &g)
{
    const float2 c = pixel_c(pm, g.x0 + g.w / 2u, g.y0 + g.h / 2u);
    if (!escape_absorbing(c.x, c.y))
        return false;
    float x = 0.0f, y = 0.0f;
#pragma unroll 8
    for (int k = 0; k < kOrderProbe; ++k)
        z_update(x, y, c.x, c.y);
    return z_bounded(x, y);
}

// Zero the per-render counters (the latched error word is kept), write the
// level-0 OLT (the axis0 x axis0 non-empty initial regions of side s0) and,
// when level 0 is queried in chunks, its per-region state.  `order` (one
// block only): regions whose probe stays bounded from slot 0 up (count[0]),
// the others from slot total - 1 down (back[0]); else in grid order.
__global__ void init_kernel(uint2 *__restrict__ olt0, uint4 *__restrict__ rst0, DevCounters *ctr,
                            uint32_t n, uint32_t s0, uint32_t axis0, uint32_t row0, uint32_t rows,
                            PixelMap pm, uint32_t order)
{
    __shared__ uint32_t s_front, s_back;
    chain_start();
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t stride = gridDim.x * blockDim.x;
    const uint32_t total = axis0 * rows;
    if (ctr != nullptr) {
        uint32_t *w = reinterpret_cast<uint32_t *>(ctr);
        const uint32_t words = (uint32_t)(sizeof(DevCounters) / sizeof(uint32_t));
        const uint32_t err_word = (uint32_t)(offsetof(DevCounters, error) / sizeof(uint32_t));
        for (uint32_t k = tid; k < words; k += stride)
            if (k != err_word)
                w[k] = (k == 0u) ? total : 0u;  // word 0 is count[0]
    }
    if (olt0 == nullptr)
        return;
    if (order) {
        if (threadIdx.x == 0) {
            s_front = 0;
            s_back = 0;
        }
        __syncthreads();  // also orders the counter words above before the totals below
    }
    for (uint32_t k = tid; k < total; k += stride) {
        const uint32_t gx = k % axis0, gy = row0 + k / axis0;
        const uint32_t x0 = gx * s0, y0 = gy * s0;
        const uint2 rec = pack_region(x0, y0, min(s0, n - x0), min(s0, n - y0));
        uint32_t slot = k;
        if (order)
            slot = region_probe(pm, unpack_region(rec)) ? atomicAdd(&s_front, 1u)
                                                        : total - 1u - atomicAdd(&s_back, 1u);
        olt0[slot] = rec;
        if (rst0 != nullptr)
            rst0[slot] = make_uint4(kNone, 0u, 0u, 0u);
    }
    if (order) {
        __syncthreads();
        if (threadIdx.x == 0 && ctr != nullptr) {
            ctr->count[0] = s_front;
            ctr->back[0] = s_back;
        }
    }
}

// ---------------------------------------------------------------------------
// Per-warp record of decided regions, flushed with one atomic per list.
// ---------------------------------------------------------------------------
template <bool BATCH>
struct WarpBatch {
    typename Rec<BATCH>::T rec;  // lane j: record of the j-th region decided
    uint32_t kind;   // KIND_*
    uint32_t nchild; // children of a splitting region
    uint32_t dwell;  // dwell of a uniform region filled later
    uint32_t sc, r;  // child side and split factor of its frame
};

// Pixel map of a region record's frame.
template <bool BATCH>
__device__ __forceinline__ PixelMap record_pm(const LevelArgs &a, const typename Rec<BATCH>::T &e)
{
    return BATCH ? a.frames[Rec<BATCH>::frame(e)].pm : a.pm;
}

// A region record from another lane.
__device__ __forceinline__ uint2 shfl_record(uint2 e, int src)
{
    return make_uint2(__shfl_sync(kFull, e.x, src), __shfl_sync(kFull, e.y, src));
}
__device__ __forceinline__ uint4 shfl_record(uint4 e, int src)
{
    return make_uint4(__shfl_sync(kFull, e.x, src), __shfl_sync(kFull, e.y, src), __shfl_sync(kFull, e.z, src),
                      0u);
}

template <bool BATCH>
__device__ __forceinline__ void flush_batch(const LevelArgs &a, WarpBatch<BATCH> &b, uint32_t lane)
{
    using R = Rec<BATCH>;
    using T = typename R::T;
    T *leaves = static_cast<T *>(a.leaves);
    T *olt_out = static_cast<T *>(a.olt_out);
    DevCounters *ctr = a.ctr;
    const unsigned lt = (1u << lane) - 1u;
    // leaves: ballot + popc gives each leaf its slot, from the front of the
    // list for the leaves whose probe stayed bounded, from the back for the
    // others
    const unsigned leaf_mask = __ballot_sync(kFull, b.kind == KIND_LEAF);
    if (leaf_mask) {
        const bool is_leaf = b.kind == KIND_LEAF;
        const bool heavy = is_leaf && region_probe(record_pm<BATCH>(a, b.rec), R::region(b.rec));
        const unsigned hm = __ballot_sync(kFull, heavy), lm = leaf_mask & ~hm;
        uint32_t hb = 0, lb = 0;
        if (lane == 0) {
            if (hm)
                hb = atomicAdd(&ctr->leaf_count, (uint32_t)__popc(hm));
            if (lm)
                lb = atomicAdd(&ctr->leaf_light, (uint32_t)__popc(lm));
        }
        hb = __shfl_sync(kFull, hb, 0);
        lb = __shfl_sync(kFull, lb, 0);
        if (is_leaf) {
            const uint32_t k = heavy ? hb + (uint32_t)__popc(hm & lt) : lb + (uint32_t)__popc(lm & lt);
            if (k < a.leaf_cap)
                leaves[heavy ? k : a.leaf_cap - 1u - k] = b.rec;
            else
                atomicOr(&ctr->error, ERR_LEAF_OVERFLOW);
        }
    }
    // large uniform regions for the fill list, as bands of rows: a warp
    // scan of the band counts, one atomicAdd, then each lane writes the
    // bands of its region
    const unsigned later_mask = __ballot_sync(kFull, b.kind == KIND_FILL_LATER);
    if (later_mask) {
        const Region g = R::region(b.rec);
        const uint32_t nb = (b.kind == KIND_FILL_LATER) ? fill_band_count(g.w, g.h) : 0u;
        uint32_t incl = nb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, incl, o);
            if (lane >= (uint32_t)o)
                incl += v;
        }
        const uint32_t total = __shfl_sync(kFull, incl, 31);
        uint32_t base = 0;
        if (lane == 0)
            base = atomicAdd(&ctr->fill_count, total);
        base = __shfl_sync(kFull, base, 0) + incl - nb;
        const uint32_t rows = fill_band_rows(g.w);
        for (uint32_t j = 0; j < nb; ++j) {
            const uint2 band = pack_region(g.x0, g.y0 + j * rows, g.w, min(rows, g.h - j * rows));
            if (base + j < a.fill_cap)
                a.fills[base + j] = make_uint4(band.x, band.y, b.dwell, R::frame(b.rec));
            else
                atomicOr(&ctr->error, ERR_OLT_OVERFLOW);
        }
    }
    // children: 32 at a time over all the regions that split, one a lane (a
    // warp scan of the counts tells a lane its region), each probed and put in
    // the next level's table, from the front or from the back
    if (__any_sync(kFull, b.nchild != 0u)) {
        uint32_t incl = b.nchild;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, incl, o);
            if (lane >= (uint32_t)o)
                incl += v;
        }
        const uint32_t total = __shfl_sync(kFull, incl, 31);
        for (uint32_t p0 = 0; p0 < total; p0 += 32u) {
            const uint32_t p = p0 + lane;
            uint32_t own = 0;  // regions (lanes) whose children all come before p
#pragma unroll
            for (uint32_t h = 16u; h >= 1u; h >>= 1)
                if (__shfl_sync(kFull, incl, (int)(own + h - 1u)) <= p)
                    own += h;
            const bool valid = p < total;
            const int src = (int)(own & 31u);
            const T rec = shfl_record(b.rec, src);
            const uint32_t j = p - (__shfl_sync(kFull, incl, src) - __shfl_sync(kFull, b.nchild, src));
            const uint32_t sc = __shfl_sync(kFull, b.sc, src), r = __shfl_sync(kFull, b.r, src);
            uint2 child = make_uint2(0u, 0u);
            bool heavy = false;
            if (valid) {
                child = child_region(R::region(rec), sc, r, j);
                heavy = region_probe(record_pm<BATCH>(a, rec), unpack_region(child));
            }
            const unsigned hm = __ballot_sync(kFull, heavy), lm = __ballot_sync(kFull, valid && !heavy);
            uint32_t hb = 0, lb = 0;
            if (lane == 0) {
                if (hm)
                    hb = atomicAdd(&ctr->count[a.level + 1], (uint32_t)__popc(hm));
                if (lm)
                    lb = atomicAdd(&ctr->back[a.level + 1], (uint32_t)__popc(lm));
            }
            hb = __shfl_sync(kFull, hb, 0);
            lb = __shfl_sync(kFull, lb, 0);
            if (valid) {
                const uint32_t k = heavy ? hb + (uint32_t)__popc(hm & lt) : lb + (uint32_t)__popc(lm & lt);
                if (k < a.out_cap) {
                    const uint32_t slot = heavy ? k : a.out_cap - 1u - k;
                    olt_out[slot] = R::child(rec, child);
                    if (a.next_chunks > 1u)
                        a.rst_out[slot] = make_uint4(kNone, 0u, 0u, 0u);
                } else {
                    atomicOr(&ctr->error, ERR_OLT_OVERFLOW);
                }
            }
        }
    }
    const unsigned fill_mask = __ballot_sync(kFull, b.kind == KIND_FILL || b.kind == KIND_FILL_LATER);
    const unsigned split_mask = __ballot_sync(kFull, b.kind == KIND_SPLIT);
    if (lane == 0) {
        if (fill_mask)
            atomicAdd(&ctr->fills[a.level], (uint32_t)__popc(fill_mask));
        if (split_mask)
            atomicAdd(&ctr->subdivs[a.level], (uint32_t)__popc(split_mask));
    }
    b.kind = KIND_NONE;
    b.nchild = 0;
}

// One chunk [k0, k1) of a large last-level region with exact perimeters:
// every dwell is computed and written; st.x / st.y collect min / max.
__device__ __forceinline__ void chunk_exact(const FView &a, const Region &g, uint32_t k0,
                                            uint32_t k1, uint4 *st, uint32_t lane,
                                            Updates &it)
{
    uint32_t dmin = kNone, dmax = 0u;
    for (uint32_t k = k0 + lane; k < k1; k += 32u) {
        uint32_t px, py;
        perimeter_pixel(g, k, px, py);
        const float2 c = pixel_c(a.pm, px, py);
        const uint32_t d = dwell(c.x, c.y, a.max_dwell, &it.spared);
        a.map[(size_t)py * a.n + px] = d;
        dmin = min(dmin, d);
        dmax = max(dmax, d);
        it += d;
    }
    dmin = __reduce_min_sync(kFull, dmin);
    dmax = __reduce_max_sync(kFull, dmax);
    if (lane == 0) {
        atomicMin(&st->x, dmin);
        atomicMax(&st->y, dmax);
    }
}

// A warp's counts of a level (COUNT mode).
__device__ __forceinline__ void count_level(const LevelArgs &a, Updates it, unsigned long long bpx, unsigned long long fpx,
                                            unsigned long long dpx, uint32_t lane)
{
    count_updates(a.ctr, &a.ctr->level_iters[a.level], &a.ctr->level_spared[a.level], it, lane);
    bpx = warp_sum_u64(bpx);
    fpx = warp_sum_u64(fpx);
    dpx = warp_sum_u64(dpx);
    if (lane == 0) {
        if (bpx)
            atomicAdd(&a.ctr->border_pixels, bpx);
        if (fpx)
            atomicAdd(&a.ctr->fill_pixels, fpx);
        if (dpx)
            atomicAdd(&a.ctr->deferred_fill_pixels, dpx);
    }
}

// ---------------------------------------------------------------------------
// Level kernel: one warp per work item (a region, or a perimeter chunk of a
// large region), NS perimeter orbits a lane.
//
// A level is bound by the latency of its items (each a few trips to L2 and a
// chain of updates) as much as by its updates, so two orbits a lane (24 warps
// an SM, up to 80 registers) are the better half wherever an item has more than 32
// pixels to give: side 18 and up, chunks of 64.  Smaller regions take one orbit
// a lane and 32 warps.  (Two for the regions of side 16 of n = 16384: 393 us
// against 371; one up to side 40, n = 1999 without chunks: 316 against 311.)
//
// Levels 0 to 3 at n = 16384 (g=16 r=4 B=16), in us: contiguous chunks, every
// orbit of the set run to max_dwell 130 / 194 / 303 / 377; perimeters spread,
// capture discs and repeats 65 / 121 / 246 / 404; two orbits a lane 67 / 106 /
// 211 / 401; cheap regions several to a ticket, chunk-major order, children
// probed one a lane 62 / 75 / 190 / 371; chunks of 64 at every level 56 / 73 /
// 186 / 371.  n = 65536 (8 levels): 6.4 -> 4.0 ms.
// ---------------------------------------------------------------------------
// CTAs an SM for one and two orbits a lane.
constexpr int kLevelMinBlocks1 = 4;
constexpr int kLevelMinBlocks2 = 3;
// Level kernels of regions up to this side take one orbit a lane.
constexpr uint32_t kLevelSide1 = 17;
// Levels that hold at most this many regions, of perimeters one CTA can take
// at a time, run one CTA per region (level_cta_kernel).  None / 512 / 2048 /
// 8192: n = 1024 71 / 66 / 60 / 60 us, n = 2048 179 / 165 / 159 / 155, n = 1999
// without chunks 278 / 195 / 195 / 201, n = 3001 385 / 386 / 370 / 370.
constexpr unsigned long long kCtaLevelRegions = 2048;
// Small regions (one orbit a lane) look for orbits that stay only where a
// region is at least this wide in the plane: nearer to the boundary proofs come
// too late to pay for the looks (level of sides 16 at n = 16384, cap 2048: 374 us
// with, 366 without; at n = 4096: 82 with, 96 without).  Whole maps without / with,
// at caps 256, 2048 and 8192: n = 4096 (sides 16, 0.0078 wide) 145 / 146, 361 / 349,
// 1010 / 883 us; n = 16384 (0.002 wide) 882 / 908, 1651 / 1654, 3830 / 3560.  At
// caps of many thousand they would pay below this line too.
// A batch's levels of whole small perimeters, and those of the persistent kernel,
// do without (64 frames of up to 8192 pixels 38.1 ms, 38.4 with proofs; persistent
// 45.3 and 45.6; 32 frames of up to 2048 3.18 and 3.10 ms, 3.47 and 3.42).
constexpr float kProveExtent = 0.004f;
// A ticket of cheap regions stands for at most kTicketMax of them, as long as
// every warp gets kTicketsPerWarp tickets (1 at most: 377 us at level 3 of n =
// 16384 and 11.0 ms at n = 65536 against 371 and 10.0; a ticket of several
// regions from the front of the table, too: 588 us).
constexpr uint32_t kTicketMax = 8;
constexpr uint32_t kTicketsPerWarp = 4;

template <bool COUNT, bool BATCH, int NS, bool PROVE>
__global__ void __launch_bounds__(256, NS == 1 ? kLevelMinBlocks1 : kLevelMinBlocks2)
    level_kernel(LevelArgs a)
{
    using R = Rec<BATCH>;
    using T = typename R::T;
    extern __shared__ uint32_t smem[];
    chain_start();
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t *stage = smem + (threadIdx.x >> 5) * kWarpStage;
    const T *olt_in = static_cast<const T *>(a.olt_in);
    // regions from the front of the table first, then those from the back
    const uint32_t front = min(a.ctr->count[a.level], a.in_cap);
    const uint32_t count = front + min(a.ctr->back[a.level], a.in_cap - front);
    if (blockIdx.x == 0 && threadIdx.x == 0 &&
        (unsigned long long)a.ctr->count[a.level] + a.ctr->back[a.level] > a.in_cap)
        atomicOr(&a.ctr->error, ERR_OLT_OVERFLOW);
    const uint32_t chunks = (NS == 1) ? 1u : a.chunks;  // one orbit a lane: small regions
    const bool query_all = !BATCH && a.split != 0u;  // no region of this level is exact

    WarpBatch<BATCH> b;
    b.rec = T();
    b.kind = KIND_NONE;
    b.nchild = 0;
    b.dwell = 0;
    b.sc = b.r = 1u;
    uint32_t j = 0;
    Updates it;
    unsigned long long bpx = 0, fpx = 0, dpx = 0;

    // The regions from the front of the table come first and are handed out one
    // item at a time: their costs differ by orders of magnitude (a uniform
    // perimeter inside the set may run to max_dwell).  Those from the back are
    // cheap; where every warp gets many of them, a ticket stands for `take`,
    // so that one round trip for the ticket and one for the records serve them
    // all.  Of either kind every region's first chunk comes before any region's
    // second: most regions that are not uniform are known by then, and their
    // other chunks end at a look at the region's state.
    const uint32_t back = count - front, heavy = front * chunks, light = back * chunks;
    const uint32_t warps = gridDim.x * (blockDim.x / 32u);
    uint32_t take = 1u;
    while (take < kTicketMax && light / (2u * take) >= kTicketsPerWarp * warps)
        take *= 2u;
    const uint32_t tickets = level_tickets(heavy, light, take);
    uint32_t todo = 0, my_c = 0, my_slot = 0;
    T mine = T();
    // a warp's first ticket is its number (counted over the CTAs first, so that
    // a short table is spread over all SMs); the counter hands out the others
    uint32_t t = blockIdx.x + gridDim.x * (threadIdx.x >> 5);
    bool fresh = true;
    for (;;) {
        if (todo == 0u) {
            if (!fresh) {
                if (lane == 0)
                    t = warps + atomicAdd(&a.ctr->work[a.level], 1u);
                t = __shfl_sync(kFull, t, 0);
            }
            if (fresh ? t >= tickets : past_tickets(t, warps, tickets))
                break;
            fresh = false;
            // lane k looks at the ticket's k-th item: its record, and, of a
            // large region, whether it is still open
            bool open;
            uint32_t li;
            if (t < heavy) {
                open = lane == 0;
                my_c = (chunks == 1u) ? 0u : t / front;
                li = t - my_c * front;
            } else {
                const uint32_t q = (t - heavy) * take + lane;
                open = lane < take && q < light;
                my_c = (chunks == 1u) ? 0u : q / back;
                li = front + (q - my_c * back);
            }
            if (open) {
                my_slot = table_slot(li, front, a.in_cap);
                if (chunks > 1u && !(COUNT && my_c == 0u) && (query_all || !a.exact_last))
                    open = reinterpret_cast<const volatile uint32_t *>(a.rst_in + my_slot)[1] == 0u;
                mine = olt_in[my_slot];
            }
            todo = __ballot_sync(kFull, open);
            continue;
        }
        const int k = __ffs((int)todo) - 1;
        todo &= todo - 1u;
        const uint32_t c = (chunks == 1u) ? 0u : __shfl_sync(kFull, my_c, k);
        const uint32_t region = (chunks == 1u) ? 0u : __shfl_sync(kFull, my_slot, k);
        const T e = shfl_record(mine, k);
        const Region g = R::region(e);
        const FView f = BATCH ? view_frame(a.frames, R::frame(e), a.level) : view_single(a);
        const bool query = f.split || !a.exact_last;
        const uint32_t P = perimeter_size(g.w, g.h);
        bool decided = false, uniform = false;
        uint32_t wv = 0;

        if (chunks == 1u) {
            decided = true;
            if (COUNT && lane == 0)
                bpx += P;
            if (query) {
                uniform = warp_perimeter_uniform<BATCH ? kQueryRoundBatch : kQueryRound, NS, PROVE>(
                    f.pm, f.max_dwell, g, lane, BATCH ? 3u : 0u, &wv, it);
            } else {
                // last level, exact perimeters staged in shared memory: a leaf
                // keeps them and the leaf kernel skips them
                uint32_t dmin = kNone, dmax = 0u;
                for (uint32_t k = lane; k < P; k += 32u) {
                    uint32_t px, py;
                    perimeter_pixel(g, k, px, py);
                    const float2 c = pixel_c(f.pm, px, py);
                    const uint32_t d = dwell(c.x, c.y, f.max_dwell, COUNT ? &it.spared : nullptr);
                    dmin = min(dmin, d);
                    dmax = max(dmax, d);
                    if (k < kWarpStage)
                        stage[k] = d;
                    else
                        f.map[(size_t)py * f.n + px] = d;  // beyond the stage: write through
                    if (COUNT)
                        it += d;
                }
                dmin = __reduce_min_sync(kFull, dmin);
                dmax = __reduce_max_sync(kFull, dmax);
                uniform = (dmin == dmax);
                wv = dmin;
                if (!uniform) {
                    const uint32_t staged = min(P, kWarpStage);
                    for (uint32_t k = lane; k < staged; k += 32u) {
                        uint32_t px, py;
                        perimeter_pixel(g, k, px, py);
                        f.map[(size_t)py * f.n + px] = stage[k];
                    }
                }
            }
        } else {
            uint4 *st = a.rst_in + region;
            if (COUNT && lane == 0 && c == 0)
                bpx += P;
            if (query) {
                const uint32_t r = chunk_query<NS>(f, g, P, c, chunks, st, BATCH ? 1u : kPollLag, lane, it);
                decided = chunk_decides(r, st, chunks, lane, uniform, wv);
            } else {
                const uint32_t CP = ceil_div_u32(P, chunks);
                const uint32_t k0 = min(P, c * CP), k1 = min(P, k0 + CP);
                if (k0 < k1)
                    chunk_exact(f, g, k0, k1, st, lane, it);
                // the warp that finishes the region's last chunk decides
                uint32_t last = 0, sx = 0, sy = 0;
                if (lane == 0) {
                    __threadfence();
                    last = (atomicAdd(&st->z, 1u) == chunks - 1u) ? 1u : 0u;
                    if (last) {
                        __threadfence();
                        sx = atomicAdd(&st->x, 0u);
                        sy = atomicAdd(&st->y, 0u);
                    }
                }
                decided = __shfl_sync(kFull, last, 0) != 0u;
                wv = __shfl_sync(kFull, sx, 0);
                uniform = wv == __shfl_sync(kFull, sy, 0);
            }
        }

        if (decided) {
            uint32_t kind;
            if (uniform) {
                const unsigned long long area = (unsigned long long)g.w * g.h;
                if (a.fills != nullptr && area > kInPlaceFillArea) {
                    kind = KIND_FILL_LATER;
                } else {
                    fill_rect(f.map, f.n, g, wv, lane, 32u);
                    kind = KIND_FILL;
                }
                if (COUNT && lane == 0) {
                    fpx += area;
                    if (kind == KIND_FILL_LATER)
                        dpx += area;
                }
            } else {
                kind = f.split ? KIND_SPLIT : KIND_LEAF;
            }
            if (lane == j) {
                b.rec = e;
                b.kind = kind;
                b.dwell = wv;
                b.sc = f.child_side;
                b.r = f.r;
                b.nchild = (kind == KIND_SPLIT) ? child_count(g, f.child_side, f.r) : 0u;
            }
            __syncwarp();
            if (++j == 32u) {
                flush_batch<BATCH>(a, b, lane);
                j = 0;
            }
        }
    }
    if (j)
        flush_batch<BATCH>(a, b, lane);
    if (COUNT)
        count_level(a, it, bpx, fpx, dpx, lane);
}

// ---------------------------------------------------------------------------
// Level kernel of a level of few regions: one CTA per region, its warps each a
// chunk of the perimeter (spread over all of it, two orbits a lane).  The
// region's query state lives in shared memory and the decision follows a
// barrier, so a region costs no ticket, no fences and no state in global
// memory, and the whole CTA fills it.
// ---------------------------------------------------------------------------
template <bool COUNT, bool BATCH>
__global__ void __launch_bounds__(256, kLevelMinBlocks2) level_cta_kernel(LevelArgs a)
{
    using R = Rec<BATCH>;
    using T = typename R::T;
    __shared__ uint4 st;
    chain_start();
    const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
    const uint32_t front = min(a.ctr->count[a.level], a.in_cap);
    const uint32_t count = front + min(a.ctr->back[a.level], a.in_cap - front);
    if (blockIdx.x == 0 && threadIdx.x == 0 &&
        (unsigned long long)a.ctr->count[a.level] + a.ctr->back[a.level] > a.in_cap)
        atomicOr(&a.ctr->error, ERR_OLT_OVERFLOW);
    Updates it;
    unsigned long long bpx = 0, fpx = 0, dpx = 0;
    for (uint32_t li = blockIdx.x; li < count; li += gridDim.x) {
        const T e = static_cast<const T *>(a.olt_in)[table_slot(li, front, a.in_cap)];
        const Region g = R::region(e);
        const FView f = BATCH ? view_frame(a.frames, R::frame(e), a.level) : view_single(a);
        const uint32_t P = perimeter_size(g.w, g.h);
        if (threadIdx.x == 0) {
            st = make_uint4(kNone, 0u, 0u, 0u);
            if (COUNT)
                bpx += P;
        }
        __syncthreads();
        chunk_query<2>(f, g, P, wib, blockDim.x / 32u, &st, 1u, lane, it);
        __syncthreads();
        const bool uniform = st.y == 0u;
        const uint32_t wv = st.x;
        uint32_t kind = f.split ? KIND_SPLIT : KIND_LEAF;
        if (uniform) {
            const unsigned long long area = (unsigned long long)g.w * g.h;
            kind = (a.fills != nullptr && area > kInPlaceFillArea) ? KIND_FILL_LATER : KIND_FILL;
            if (kind == KIND_FILL)
                fill_rect(f.map, f.n, g, wv, threadIdx.x, blockDim.x);
            if (COUNT && threadIdx.x == 0) {
                fpx += area;
                if (kind == KIND_FILL_LATER)
                    dpx += area;
            }
        }
        if (wib == 0) {
            WarpBatch<BATCH> b;
            b.rec = e;
            b.kind = lane == 0 ? kind : KIND_NONE;
            b.dwell = wv;
            b.sc = f.child_side;
            b.r = f.r;
            b.nchild = (lane == 0 && kind == KIND_SPLIT) ? child_count(g, f.child_side, f.r) : 0u;
            flush_batch<BATCH>(a, b, lane);
        }
        __syncthreads();  // st is free for the next region
    }
    if (COUNT)
        count_level(a, it, bpx, fpx, dpx, lane);
}

// ---------------------------------------------------------------------------
// Fill kernel: the bands of the large uniform regions (at most kFillBandPx
// pixels each), one band per warp item, 128-bit stores; pure HBM writes.
// ---------------------------------------------------------------------------
template <bool BATCH>
__global__ void __launch_bounds__(256) fill_kernel(FillArgs f)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t nfill = min(f.ctr->fill_count, f.fill_cap);
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t fi = warp; fi < nfill; fi += nwarps) {
        const uint4 e = f.fills[fi];
        const Region g = unpack_region(make_uint2(e.x, e.y));
        if (BATCH) {
            const FrameDesc &d = f.frames[e.w];
            fill_band_warp(d.map, d.n, g, e.z, lane);
        } else {
            fill_band_warp(f.map, f.n, g, e.z, lane);
        }
    }
}

// ---------------------------------------------------------------------------
// Tiled leaf kernel (ASK_FLAG_LEAF_TILED): (leaf, tile) items with block_x x
// block_y tiles, one thread per pixel; persistent grid, warps walk the item
// sequence on their own.
// ---------------------------------------------------------------------------
template <bool COUNT>
__global__ void __launch_bounds__(1024) leaf_kernel(LeafArgs a, uint32_t leaf_cap, uint32_t tiles_x,
                                                    uint32_t tiles_per_leaf)
{
    uint32_t front, nleaves;
    leaf_extent(a.ctr, leaf_cap, front, nleaves);
    const unsigned long long total = (unsigned long long)nleaves * tiles_per_leaf;
    Updates it;
    unsigned long long lpx = 0;
    for (unsigned long long item = blockIdx.x; item < total; item += gridDim.x) {
        const uint32_t leaf = (uint32_t)(item / tiles_per_leaf);
        const uint32_t t = (uint32_t)(item - (unsigned long long)leaf * tiles_per_leaf);
        const Region g = unpack_region(static_cast<const uint2 *>(a.leaves)[table_slot(leaf, front, leaf_cap)]);
        const uint32_t ty = t / tiles_x, tx = t - ty * tiles_x;
        const uint32_t px = g.x0 + tx * blockDim.x + threadIdx.x;
        const uint32_t py = g.y0 + ty * blockDim.y + threadIdx.y;
        if (px < g.x0 + g.w && py < g.y0 + g.h && !(a.skip_perimeter && on_perimeter(g, px, py))) {
            const float2 c = pixel_c(a.pm, px, py);
            const uint32_t d = dwell<false>(c.x, c.y, a.max_dwell);
            a.map[(size_t)py * a.n + px] = d;
            if (COUNT) {
                it += d;
                ++lpx;
            }
        }
    }
    if (COUNT) {
        const uint32_t lane = (threadIdx.x + threadIdx.y * blockDim.x) % 32u;
        count_updates(a.ctr, &a.ctr->leaf_iters, &a.ctr->leaf_spared, it, lane);
        lpx = warp_sum_u64(lpx);
        if (lane == 0u && lpx)
            atomicAdd(&a.ctr->leaf_pixels, lpx);
    }
}

// ---------------------------------------------------------------------------
// Leaf kernel (default): a coherent first pass over fresh pixels, then lane
// refill for the orbits that survive it.
//
// Leaf pixels lie near the set's boundary: their dwells run from a handful
// of updates to max_dwell side by side (at n = 16384 the median leaf pixel
// escapes after 19 updates, 71% within 32, while the 5% that reach max_dwell
// hold two thirds of the updates).  A warp that owned 32 fixed pixels would
// idle most lanes while one orbit runs on, so each warp takes leaves from a
// device counter and works in two stages:
//  * pre-pass: 64 fresh pixels at a time, two per lane, all lanes in
//    lockstep, run their first kPrePass updates in unchecked blocks of
//    kPreBlock with one test per block (see dwell()).  An orbit that escapes
//    there is resolved on the spot by a binary search over its last block
//    and written; the others are pushed, with their state, onto the warp's
//    ring of survivors in shared memory.  Most pixels end here, with no
//    per-pixel bookkeeping beyond the lane they run on;
//  * refill loop over the survivors: each lane carries two orbits; every
//    round each orbit runs two unchecked blocks of kLeafUnroll updates; an
//    orbit that escaped (or has less than a block left) waits at the block's
//    start until kRefillSlots slots wait or are idle; then the waiting ones
//    go to the warp's park buffer and the free slots take the next survivors
//    from the ring (the pre-pass tops the ring up when it runs short).  An
//    orbit that reaches max_dwell at a block's end, or repeats an earlier
//    state, is written there and then;
//  * when 32 orbits are parked, the warp finishes them together, one per
//    lane: a binary search over the parked block finds the exact escape (the
//    block's midpoint state is parked too, so the first halving costs one
//    test; then unchecked quarter, eighth, ... blocks and one test each, the
//    same number of steps on every lane), and the dwells are written;
//  * the leaves are taken in the order of the list, whose front holds the
//    leaves whose centre orbit the level kernel's probe found bounded (most
//    long orbits), so the warps end on short orbits; once the list has run
//    out and a warp's orbits fit in one slot per lane, slot 1 folds into
//    slot 0 and the last rounds update one orbit per lane.
//
// What bounds it is issue slots (a packed update pair holds the dispatch port
// as long as two scalar updates): at n = 16384 (g=16 r=4 B=16) it issues or
// dispatches on about 92% of its active cycles and the FP32 pipe is busy on
// 64%.  So what it saves is instructions around the updates.  One pixel a lane
// in the pre-pass, parking and refilling every round, and the cursor and the
// limits in registers (48 a thread, spilled) took 1.17-1.20 ms, this form
// 0.93-0.94 (0.97 without the test for a repeated state); n = 65536 (g=32 r=2
// B=16) 7.5 -> 6.0 ms; 64 mixed frames in a batch 33.5 -> 29.6 ms.
// ---------------------------------------------------------------------------
// The leaf kernel over the leaf list of a launch chain.  Each lane of the
// refill loop carries two independent orbits, so one round's bookkeeping
// (votes, refills, parking) serves two blocks of updates, and the two update
// chains interleave.  Parked orbits and ring entries remember their frame.
template <bool COUNT, bool BATCH>
__global__ void __launch_bounds__(kRefillWarps * 32, kRefillMinBlocks) leaf_refill_kernel(LeafArgs a)
{
    __shared__ WarpLeaf<BATCH> shared[kRefillWarps];
    __shared__ uint3 extent;                           // front, leaves, item shift (LeafList)
    chain_start();
    const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        uint32_t front, total;
        leaf_extent(a.ctr, a.leaf_cap, front, total);
        const uint32_t warps = gridDim.x * (uint32_t)kRefillWarps;
        const uint32_t shift = leaf_item_shift(total, a.side, warps);
        if (!leaf_items_fit(total, shift, warps)) {
            atomicOr(&a.ctr->error, ERR_LEAF_OVERFLOW);
            total = 0;
        }
        extent = make_uint3(front, total, shift);
    }
    __syncthreads();
    if (a.fills != nullptr && wib == kRefillWarps - 1u)
        drain_fills<BATCH>(a, lane);  // the CTA's fill warp
    WarpLeaf<BATCH> &w = shared[wib];
    WarpFill f;
    f.parked = f.ring_h = f.ring_n = 0;

    LeafList<BATCH> src;
    src.leaves = static_cast<const typename Rec<BATCH>::T *>(a.leaves);
    src.cap = a.leaf_cap;
    src.extent = &extent;
    uint32_t srcst = SRC_MORE;
    cursor_reset(w.cursor, lane);
    Updates it;
    unsigned long long lpx = 0;
    PrePassFeed<COUNT, BATCH, LeafList<BATCH>> feed{src};
    // a small batch: pre-passes only, the survivors to the pool while it has room
    if (BATCH && a.pool != nullptr)
        do
            feed(a, srcst, w, f, lane, it, lpx);
        while (pool_survivors<BATCH>(a, w, f, lane) && srcst == SRC_MORE);
    if (f.ring_n != 0u || srcst == SRC_MORE)
        run_orbits<COUNT, BATCH>(a, feed, srcst, w, f, lane, it, lpx);
    if (a.fills != nullptr)
        drain_fills<BATCH>(a, lane);
    finish_orbits<COUNT, BATCH>(a, w, f, lane, it, lpx);
}

// ---------------------------------------------------------------------------
// Second kernel of a small batch's leaves: the pooled survivors, dealt evenly.
//
// In the leaf kernel of a small batch a warp that took a few heavy leaves runs
// on long after the others; pooled, its orbits are dealt to all warps, 32 at a
// time, and to no more warps than they fill (kPoolPerWarp each, spread over the
// schedulers), since a round costs the same for 5 lanes as for 64.  12 frames
// of up to 1024 pixels as a graph: 456 -> 364 us (leaf kernel 265 us; 77 + 117
// with the pool).  Single frames keep their survivors: their leaves are alike
// enough, and the second kernel cost more than it gave (n = 3001 362 -> 379 us,
// n = 1024 60 -> 64 us, n = 4096 354 -> 344 us).
// ---------------------------------------------------------------------------
constexpr uint32_t kPoolPerWarp = 64;
template <bool COUNT>
__global__ void __launch_bounds__(kRefillWarps * 32, kRefillMinBlocks) pool_kernel(LeafArgs a, uint32_t resident)
{
    __shared__ WarpLeaf<true> shared[kRefillWarps];
    chain_start();
    const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
    const uint32_t total = min(a.ctr->pool_count, a.pool_cap);
    // active warps per CTA, rotated from CTA to CTA of an SM so that they
    // spread over its schedulers
    const uint32_t per_cta = min((uint32_t)kRefillWarps,
                                 (total + kPoolPerWarp * gridDim.x - 1u) / (kPoolPerWarp * gridDim.x));
    const uint32_t rank = (wib + blockIdx.x * resident / gridDim.x) % (uint32_t)kRefillWarps;
    if (rank >= per_cta)
        return;
    WarpLeaf<true> &w = shared[wib];
    WarpFill f;
    f.parked = f.ring_h = f.ring_n = 0;
    PoolFeed feed;
    feed.total = total;
    feed.next = kPoolTake * (blockIdx.x + gridDim.x * rank);
    feed.first_end = kPoolTake * gridDim.x * per_cta;
    Updates it;
    unsigned long long lpx = 0;
    run_orbits<COUNT, true>(a, feed, SRC_MORE, w, f, lane, it, lpx);
    finish_orbits<COUNT, true>(a, w, f, lane, it, lpx);
}

// Level-0 records and counters of a batch: block f writes frame f's
// axis0 x axis0 initial regions at its offset; block 0 zeroes the counters.
__global__ void init_batch_kernel(uint4 *__restrict__ olt0, uint4 *__restrict__ rst0,
                                  DevCounters *ctr, const FrameDesc *frames, uint32_t total0)
{
    chain_start();
    const uint32_t f = blockIdx.x;
    if (f == 0) {
        uint32_t *w = reinterpret_cast<uint32_t *>(ctr);
        const uint32_t words = (uint32_t)(sizeof(DevCounters) / sizeof(uint32_t));
        const uint32_t err_word = (uint32_t)(offsetof(DevCounters, error) / sizeof(uint32_t));
        for (uint32_t k = threadIdx.x; k < words; k += blockDim.x)
            if (k != err_word)
                w[k] = (k == 0u) ? total0 : 0u;  // word 0 is count[0]
    }
    const FrameDesc &d = frames[f];
    const uint32_t per = d.axis0 * d.axis0;
    for (uint32_t k = threadIdx.x; k < per; k += blockDim.x) {
        const uint32_t gx = k % d.axis0, gy = k / d.axis0;
        const uint32_t x0 = gx * d.s0, y0 = gy * d.s0;
        const uint2 rec = pack_region(x0, y0, min(d.s0, d.n - x0), min(d.s0, d.n - y0));
        olt0[d.olt0_offset + k] = make_uint4(rec.x, rec.y, f, 0u);
        if (rst0 != nullptr)
            rst0[d.olt0_offset + k] = make_uint4(kNone, 0u, 0u, 0u);
    }
}

}  // namespace

cudaError_t launch_exhaustive(uint32_t *map, uint32_t n, PixelMap pm, uint32_t max_dwell,
                              uint32_t bx, uint32_t by, bool count, DevCounters *ctr,
                              cudaStream_t s)
{
    const uint32_t tiles_x = (n + bx - 1) / bx, tiles_y = (n + by - 1) / by;
    const dim3 block(bx, by);
    const unsigned long long tiles = (unsigned long long)tiles_x * tiles_y;
    if (tiles > 0x7fffffffull)
        return cudaErrorInvalidConfiguration;
    if (count)
        exhaustive_kernel<true><<<(unsigned)tiles, block, 0, s>>>(map, n, pm, max_dwell, tiles_x, ctr);
    else
        exhaustive_kernel<false><<<(unsigned)tiles, block, 0, s>>>(map, n, pm, max_dwell, tiles_x, ctr);
    return cudaGetLastError();
}

cudaError_t launch_init(uint2 *olt0, uint4 *rst0, DevCounters *ctr, uint32_t n, uint32_t s0,
                        uint32_t axis0, uint32_t row0, uint32_t rows, cudaStream_t s,
                        const PixelMap *order)
{
    const uint32_t total = axis0 * rows;
    if (order != nullptr && olt0 != nullptr && total <= kInitOrderMax) {
        init_kernel<<<1, 1024, 0, s>>>(olt0, rst0, ctr, n, s0, axis0, row0, rows, *order, 1u);
        return cudaGetLastError();
    }
    uint32_t blocks = (total + 255u) / 256u;
    if (blocks < 1)
        blocks = 1;
    if (blocks > 4096)
        blocks = 4096;
    init_kernel<<<blocks, 256, 0, s>>>(olt0, rst0, ctr, n, s0, axis0, row0, rows, PixelMap{}, 0u);
    return cudaGetLastError();
}

template <bool COUNT, bool BATCH, int NS, bool PROVE>
static cudaError_t level_launch(const LevelArgs &a, int sms, cudaStream_t s)
{
    const size_t stage = (size_t)(256 / 32) * kWarpStage * sizeof(uint32_t);
    const size_t smem = a.exact_last ? stage : 0u;
    static PerDevice plain, staged;
    // no more CTAs than the level can have items for, but one an SM as long as
    // there is an item for each
    const unsigned long long items = a.bound * a.chunks;
    const unsigned long long most = std::max((items + 7u) / 8u, std::min(items, (unsigned long long)sms));
    int grid = resident_ctas(level_kernel<COUNT, BATCH, NS, PROVE>, 256, smem, a.exact_last ? &staged : &plain) * sms;
    if (most < (unsigned long long)grid)
        grid = most ? (int)most : 1;
    return launch_chained(level_kernel<COUNT, BATCH, NS, PROVE>, grid, 256, smem, s, a);
}

template <bool COUNT, bool BATCH>
static cudaError_t level_launch_sized(const LevelArgs &a, int sms, cudaStream_t s)
{
    const bool query_all = !a.exact_last || (!BATCH && a.split != 0u);
    if (a.bound <= kCtaLevelRegions && query_all && (a.chunks <= 8u || a.rst_in == nullptr))
        return launch_chained(level_cta_kernel<COUNT, BATCH>, std::max(1, (int)a.bound),
                              32 * (int)std::min(8u, std::max(1u, (4u * a.side + 63u) / 64u)), 0, s, a);
    if (a.chunks > 1u || (!BATCH && a.side > kLevelSide1))
        return level_launch<COUNT, BATCH, 2, true>(a, sms, s);
    if constexpr (!BATCH)
        if ((float)a.side * std::max(a.pm.dx, a.pm.dy) >= kProveExtent)
            return level_launch<COUNT, BATCH, 1, true>(a, sms, s);
    return level_launch<COUNT, BATCH, 1, false>(a, sms, s);
}

cudaError_t launch_level(const LevelArgs &a, bool count, bool batch, int sms, cudaStream_t s)
{
    if (batch)
        return count ? level_launch_sized<true, true>(a, sms, s) : level_launch_sized<false, true>(a, sms, s);
    return count ? level_launch_sized<true, false>(a, sms, s) : level_launch_sized<false, false>(a, sms, s);
}

cudaError_t launch_fill(const FillArgs &f, bool batch, int sms, cudaStream_t s)
{
    if (batch) {
        const int grid = resident_ctas(fill_kernel<true>, 256, 0) * sms;
        fill_kernel<true><<<grid, 256, 0, s>>>(f);
    } else {
        const int grid = resident_ctas(fill_kernel<false>, 256, 0) * sms;
        fill_kernel<false><<<grid, 256, 0, s>>>(f);
    }
    return cudaGetLastError();
}

cudaError_t launch_init_batch(uint4 *olt0, uint4 *rst0, DevCounters *ctr, const FrameDesc *frames,
                              uint32_t nframes, uint32_t total0, cudaStream_t s)
{
    init_batch_kernel<<<nframes, 256, 0, s>>>(olt0, rst0, ctr, frames, total0);
    return cudaGetLastError();
}

template <bool COUNT, bool BATCH>
static cudaError_t refill_launch(const LeafArgs &a, int sms, cudaStream_t s)
{
    const int threads = kRefillWarps * 32;
    // no more CTAs than the leaves can have pre-passes for
    const unsigned long long most = a.bound * a.side * a.side / (64u * kRefillWarps) + 1u;
    static PerDevice known, known_pool;
    const int resident = resident_ctas(leaf_refill_kernel<COUNT, BATCH>, threads, 0, &known);
    const int grid = (int)std::min<unsigned long long>(most, (unsigned long long)(resident * sms));
    const cudaError_t e = launch_chained(leaf_refill_kernel<COUNT, BATCH>, grid, threads, 0, s, a);
    if (!BATCH || e != cudaSuccess || a.pool == nullptr)
        return e;
    const int pooled = resident_ctas(pool_kernel<COUNT>, threads, 0, &known_pool);
    const int pgrid = (int)std::min<unsigned long long>(most, (unsigned long long)(pooled * sms));
    return launch_chained(pool_kernel<COUNT>, pgrid, threads, 0, s, a, (uint32_t)pooled);
}

cudaError_t launch_leaf(const LeafArgs &a, uint32_t bx, uint32_t by, bool count, bool tiled,
                        bool batch, int sms, cudaStream_t s)
{
    if (batch) {
        if (tiled)
            return cudaErrorInvalidValue;
        return count ? refill_launch<true, true>(a, sms, s) : refill_launch<false, true>(a, sms, s);
    }
    if (!tiled)
        return count ? refill_launch<true, false>(a, sms, s) : refill_launch<false, false>(a, sms, s);
    const uint32_t tiles_x = (a.side + bx - 1) / bx, tiles_y = (a.side + by - 1) / by;
    const dim3 block(bx, by);
    const int threads = (int)(bx * by);
    if (count) {
        const int grid = resident_ctas(leaf_kernel<true>, threads, 0) * sms;
        leaf_kernel<true><<<grid, block, 0, s>>>(a, a.leaf_cap, tiles_x, tiles_x * tiles_y);
    } else {
        const int grid = resident_ctas(leaf_kernel<false>, threads, 0) * sms;
        leaf_kernel<false><<<grid, block, 0, s>>>(a, a.leaf_cap, tiles_x, tiles_x * tiles_y);
    }
    return cudaGetLastError();
}

}  // namespace ask
