// ask_device.cuh -- device helpers shared by the exhaustive, ASK and CDP2
// kernels: the per-pixel dwell, the pixel -> c mapping, region records,
// perimeter enumeration and vectorised fills.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "ask_internal.h"

namespace ask {

// z-updates of a counting render.  counted: as far as each orbit was followed,
// an orbit proven to stay with max_dwell; spared: those of them that were not
// run, from the proof to max_dwell.
struct Updates {
    unsigned long long counted = 0, spared = 0;
    __device__ __forceinline__ void operator+=(uint32_t d) { counted += d; }
};

// Add a whole warp's updates to the render's counters and to those of a part
// of it (NULL: none).
__device__ __forceinline__ void count_updates(DevCounters *ctr, unsigned long long *part,
                                              unsigned long long *part_spared, Updates it, uint32_t lane)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        it.counted += __shfl_xor_sync(0xffffffffu, it.counted, o);
        it.spared += __shfl_xor_sync(0xffffffffu, it.spared, o);
    }
    if (lane != 0)
        return;
    if (it.counted) {
        atomicAdd(&ctr->iterations, it.counted);
        if (part)
            atomicAdd(part, it.counted);
    }
    if (it.spared) {
        atomicAdd(&ctr->spared, it.spared);
        if (part)
            atomicAdd(part_spared, it.spared);
    }
}

// Updates per unchecked block of the dwell loops: the first and the others of
// the loop with proofs, and those of the plain loop (see dwell()).
constexpr int kFirstBlock = 16;
constexpr int kUnroll = 32;
constexpr int kPlainBlock = 16;

// |c|^2 bound below which escape is absorbing in float arithmetic (see dwell()).
constexpr float kAbsorbR2 = 3.999f;

__device__ __forceinline__ float2 pixel_c(const PixelMap &pm, uint32_t px, uint32_t py)
{
    return make_float2(__fmaf_rn(__uint2float_rn(px), pm.dx, pm.re_min),
                       __fmaf_rn(__uint2float_rn(py), pm.dy, pm.im_min));
}

// One update z <- z^2 + c, each operation rounded once (the _rn intrinsics
// are never fused or reassociated by the compiler):
//   zr' = fma(zr, zr, fma(-zi, zi, cr)),  zi' = fma(zr + zr, zi, ci).
__device__ __forceinline__ void z_update(float &x, float &y, float cr, float ci)
{
    const float t = __fmaf_rn(-y, y, cr);
    const float nx = __fmaf_rn(x, x, t);
    const float ny = __fmaf_rn(__fadd_rn(x, x), y, ci);
    x = nx;
    y = ny;
}

// Two orbits side by side: one update of each, the same operations and bits
// as z_update.  The real part stays scalar (its inner operation takes a sign
// on an operand, which the packed form lacks); the doubling and the imaginary
// part are packed operations on register pairs.  A packed operation takes the
// FP32 pipe and the dispatch port twice as long as a scalar one, so the gain is
// small: a loop of nothing but updates runs 8.0e12 updates/s scalar and
// 8.3e12 this way (of the pipe's 10.07e12); the leaf kernel at n = 16384 takes
// 1.09 ms scalar, 0.95 with all but the inner operation packed, 0.94 this way.
using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}

__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ void z_update2(f32x2 &x, f32x2 &y, f32x2 cr, f32x2 ci)
{
    float x0, x1, y0, y1, c0, c1;
    unpack2(x, x0, x1);
    unpack2(y, y0, y1);
    unpack2(cr, c0, c1);
    const f32x2 nx = pack2(__fmaf_rn(x0, x0, __fmaf_rn(-y0, y0, c0)),
                           __fmaf_rn(x1, x1, __fmaf_rn(-y1, y1, c1)));
    y = fma2(add2(x, x), y, ci);
    x = nx;
}

// The escape test of the current state: |z|^2 = fma(zr, zr, zi*zi) < 4.
__device__ __forceinline__ bool z_bounded(float x, float y)
{
    return __fmaf_rn(x, x, __fmul_rn(y, y)) < 4.0f;
}

// Escape is absorbing when |c| < 2 - 2.4e-4, i.e. fma(cr, cr, ci*ci) < 3.999:
// if the rounded |z_j|^2 >= 4 then the exact |z_j|^2 > 4 - 4e-7, so the exact
// |z_j^2 + c| > 2 + 2.3e-4, and the rounding of one update (a few ulps of
// |z|^2) cannot take it back below 2; by induction |z| keeps growing until it
// overflows, and an inf or NaN state also fails the test "|z|^2 < 4".  So for
// such c, a state that passes the test proves that every earlier state passed.
__device__ __forceinline__ bool escape_absorbing(float cr, float ci)
{
    return __fmaf_rn(cr, cr, __fmul_rn(ci, ci)) < kAbsorbR2;
}

__device__ __forceinline__ float sqrt_approx(float v)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// Principal square root of u + iv, near enough (its error is bounded by what
// capture_disc computes with the result, not assumed).
__device__ __forceinline__ float2 csqrt_near(float u, float v)
{
    const float m = sqrt_approx(__fmaf_rn(u, u, __fmul_rn(v, v)));
    const float h = sqrt_approx(0.5f * (m + fabsf(u)));
    const float k = __fdividef(0.5f * fabsf(v), h);
    return u >= 0.0f ? make_float2(h, copysignf(k, v)) : make_float2(k, copysignf(h, v));
}

// A disc around a that the iteration maps into itself: an orbit that enters
// it never escapes, however many updates follow, so its dwell is max_dwell.
// r2 is the squared radius, negative when no disc was found.
//
// One disc around a point a near the attracting fixed point: for |z - a| <= r
// a float update gives z' = z^2 + c + e with
//   |z' - a| <= |z - a| |z + a| + |a^2 + c - a| + |e|
//            <= r (2|a| + r) + q,
// where q bounds the residual |a^2 + c - a| (computed, plus its own rounding,
// 5e-7) and the update's rounding (|z| <= 1/2 there: 1.4e-7).  With D = 1 -
// 2|a| and r = D / 2 this is at most r if D^2 / 4 >= q; the constant 1.2e-6
// covers both roundings and that of D.  The bound holds for whatever a was
// computed; a poor one only makes the residual large and the disc fail.
//
// Two discs around b and b' = -1 - b near the attracting 2-cycle, of radii r
// and r1 = r (2|b| + r) + q, mapped into one another if r1 (2|b'| + r1) + q <=
// r; both discs lie in |z| < 1.9, where an update rounds by less than 1e-6.
// b is the point of the cycle nearer to the orbit's present state (x, y).
__device__ __forceinline__ void capture_disc(float cr, float ci, float x, float y, float &ax, float &ay,
                                             float &r2)
{
    r2 = -1.0f;
    const float2 s = csqrt_near(1.0f - 4.0f * cr, -4.0f * ci);
    ax = 0.5f * (1.0f - s.x);
    ay = -0.5f * s.y;
    const float D = 1.0f - 2.0f * sqrt_approx(__fmaf_rn(ax, ax, __fmul_rn(ay, ay)));
    if (D > 0.0f) {
        const float qx = __fmaf_rn(ax, ax, cr) - __fmaf_rn(ay, ay, ax);
        const float qy = __fmaf_rn(ax + ax, ay, ci) - ay;
        if (0.25f * D * D >= fabsf(qx) + fabsf(qy) + 1.2e-6f)
            r2 = 0.24999f * D * D;
        return;
    }
    const float2 q = csqrt_near(-3.0f - 4.0f * cr, -4.0f * ci);
    float bx = 0.5f * (q.x - 1.0f), by = 0.5f * q.y;
    float ex = -1.0f - bx, ey = -by;
    const float db = __fmaf_rn(x - bx, x - bx, __fmul_rn(y - by, y - by));
    const float de = __fmaf_rn(x - ex, x - ex, __fmul_rn(y - ey, y - ey));
    if (de < db) {
        const float tx = bx, ty = by;
        bx = ex;
        by = ey;
        ex = tx;
        ey = ty;
    }
    ax = bx;
    ay = by;
    const float A = 2.0f * sqrt_approx(__fmaf_rn(bx, bx, __fmul_rn(by, by)));
    const float B = 2.0f * sqrt_approx(__fmaf_rn(ex, ex, __fmul_rn(ey, ey)));
    const float r = __fdividef(0.4f * (1.0f - A * B), B + A * A + 0.5f);
    // residuals b^2 + c - b' and b'^2 + c - b, with their roundings
    const float q1 = fabsf(__fmaf_rn(bx, bx, cr) - __fmaf_rn(by, by, ex)) +
                     fabsf(__fmaf_rn(bx + bx, by, ci) - ey) + 3e-6f;
    const float q2 = fabsf(__fmaf_rn(ex, ex, cr) - __fmaf_rn(ey, ey, bx)) +
                     fabsf(__fmaf_rn(ex + ex, ey, ci) - by) + 3e-6f;
    const float r1 = r * (A + r) + q1;
    if (r > 0.0f && r1 * (B + r1) + q2 <= 0.9999f * r && 0.5f * A + r < 1.9f && 0.5f * B + r1 < 1.9f)
        r2 = 0.9999f * r * r;
}

// Whether c can have a capture disc at all: it lies in the main cardioid or in
// the period-2 disc (up to rounding; a filter that saves the others the work:
// n = 3001 at zoom 60 408 -> 393 us, n = 1999 at zoom 300 311 -> 284 us).
__device__ __forceinline__ bool may_capture(float cr, float ci)
{
    const float u = cr - 0.25f, i2 = ci * ci, q = __fmaf_rn(u, u, i2), v = cr + 1.0f;
    return q * (q + u) < 0.25f * i2 || __fmaf_rn(v, v, i2) < 0.0625f;
}

// Whether the orbit of c, at state (x, y), is in its capture disc.
__device__ __forceinline__ bool captured(float cr, float ci, float x, float y)
{
    float ax, ay, r2;
    capture_disc(cr, ci, x, y, ax, ay, r2);
    const float ux = x - ax, uy = y - ay;
    return __fmaf_rn(ux, ux, __fmul_rn(uy, uy)) < r2;
}

// Dwell of an orbit whose state (x, y) at count d passed the test and whose
// state K updates later failed, where escape is absorbing: halving the gap
// finds the first failing state (K - 1 updates, log2(K) tests).
template <uint32_t K>
__device__ __forceinline__ uint32_t dwell_in_block(float x, float y, float cr, float ci, uint32_t d)
{
#pragma unroll
    for (uint32_t h = K / 2u; h >= 1u; h >>= 1) {
        float tx = x, ty = y;
#pragma unroll
        for (uint32_t k = 0; k < h; ++k)
            z_update(tx, ty, cr, ci);
        if (z_bounded(tx, ty)) {
            x = tx;
            y = ty;
            d += h;
        }
    }
    return d + 1u;
}

// Dwell of c (paper Sec. 6): the number of updates z <- z^2 + c, from z = 0,
// made while |z|^2 < 4, at most max_dwell.
//
// Where escape is absorbing, updates run in blocks with a single test on the
// block's last state: 3 FFMA + 1 FADD per update, the test amortised over the
// block; a block whose last state fails the test holds the dwell, which is
// found behind the loop, so that the lanes of a warp do it together, and is
// exactly the stepwise count.  Other points, and the tail below max_dwell, take
// the tested loop.
//
// Two loops do this.  A warp with a point that may have a capture disc takes
// blocks of kFirstBlock and then kUnroll, and every two of them ends the orbits
// that would stay for ever: those that repeat a saved state and, at doubling
// counts, when the state is saved anew, those that have entered their disc.  A
// warp with none takes the plain loop (blocks of kPlainBlock, replayed by
// tested updates): the proofs would cost a zoom outside the two largest
// components 3-6%.  The exhaustive kernel at n = 16384, cap 2048, over the whole
// set: 28.8 ms with every orbit of the set run to the cap, 6.28 this way; n =
// 4096 1.86 -> 0.46 ms; n = 2048 at zoom 400, cap 1024: 0.259 -> 0.258.
// PROVE = false leaves the first loop out: for the pixels of leaves (tiled, SBR,
// MBR) and the regions CDP2 would make leaves, whose orbits lie along the
// boundary, where proofs come late or never (n = 16384, cap 2048: ASK-MBR 3.80
// ms with proofs, 3.58 without; tiled leaves 2.55 -> 2.41; DP-MBR 5.87 -> 5.60).
// CDP2's own leaves keep them: n = 1024, B = 32 0.410 ms without, 0.296 with.
// `spared` (or NULL) gains the updates that a proof saved.
template <bool PROVE = true>
__device__ __forceinline__ uint32_t dwell(float cr, float ci, uint32_t max_dwell,
                                          unsigned long long *spared = nullptr)
{
    float x = 0.0f, y = 0.0f;
    uint32_t d = 0;
    if (escape_absorbing(cr, ci)) {
        const bool may = PROVE && may_capture(cr, ci);
        if (PROVE && __any_sync(__activemask(), may)) {  // (either loop gives the same dwell)
            float bx = 0.0f, by = 0.0f, tx = 0.0f, ty = 0.0f;
            uint32_t age = 0;
            bool esc = false, in = false;
            if (max_dwell >= (uint32_t)kFirstBlock) {
#pragma unroll
                for (int k = 0; k < kFirstBlock; ++k)
                    z_update(tx, ty, cr, ci);
                if (!z_bounded(tx, ty))
                    return dwell_in_block<kFirstBlock>(0.0f, 0.0f, cr, ci, 0u);
                x = bx = tx;
                y = by = ty;
                d = (uint32_t)kFirstBlock;
            }
            while (max_dwell - d >= (uint32_t)kUnroll) {
                tx = x;
                ty = y;
#pragma unroll
                for (int k = 0; k < kUnroll; ++k)
                    z_update(tx, ty, cr, ci);
                esc = !z_bounded(tx, ty);
                if (esc)
                    break;
                x = tx;
                y = ty;
                d += (uint32_t)kUnroll;
                age += (uint32_t)kUnroll;
                if (age % (2u * kUnroll) == 0u) {
                    in = x == bx && y == by;
                    if (!in && (age & (age - 1u)) == 0u) {
                        in = may && captured(cr, ci, x, y);
                        bx = x;
                        by = y;
                    }
                    if (in)
                        break;
                }
            }
            if (in) {
                if (spared)
                    *spared += max_dwell - d;
                return max_dwell;
            }
            if (esc)
                return dwell_in_block<kUnroll>(x, y, cr, ci, d);
            // (less than a block is left: half a block before the tested
            // updates.  Without, low caps are slower than with no proofs:
            // CDP2, n = 2048, cap 72, leaves of 64 117 us against 92, 97 so)
            if (max_dwell - d >= (uint32_t)kFirstBlock) {
                tx = x;
                ty = y;
#pragma unroll
                for (int k = 0; k < kFirstBlock; ++k)
                    z_update(tx, ty, cr, ci);
                if (!z_bounded(tx, ty))
                    return dwell_in_block<kFirstBlock>(x, y, cr, ci, d);
                x = tx;
                y = ty;
                d += (uint32_t)kFirstBlock;
            }
        } else {
            while (max_dwell - d >= (uint32_t)kPlainBlock) {
                const float sx = x, sy = y;
#pragma unroll
                for (int k = 0; k < kPlainBlock; ++k)
                    z_update(x, y, cr, ci);
                if (!z_bounded(x, y)) {
                    x = sx;
                    y = sy;
                    break;
                }
                d += (uint32_t)kPlainBlock;
            }
        }
    }
    while (d < max_dwell && z_bounded(x, y)) {
        z_update(x, y, cr, ci);
        ++d;
    }
    return d;
}

// The same by tested updates alone (perimeter groups with points of |c| near
// 2; out of line, off the queries' way).
static __device__ __noinline__ uint32_t dwell_tested(float cr, float ci, uint32_t limit)
{
    float x = 0.0f, y = 0.0f;
    uint32_t d = 0;
    while (d < limit && z_bounded(x, y)) {
        z_update(x, y, cr, ci);
        ++d;
    }
    return d;
}

// Resumable orbit of one point, for perimeter queries that stop early.
struct Orbit {
    float x, y, cr, ci;
    uint32_t d;     // updates made; every state before z_d passed the test
    bool fast;      // escape is absorbing for this c
};

__device__ __forceinline__ Orbit orbit_start(float2 c)
{
    Orbit o;
    o.x = 0.0f;
    o.y = 0.0f;
    o.cr = c.x;
    o.ci = c.y;
    o.d = 0;
    o.fast = escape_absorbing(c.x, c.y);
    return o;
}

// Outcome of one round of an orbit.
enum : uint32_t {
    ORBIT_RUN = 0,   // every state so far passed; more rounds to go
    ORBIT_DONE = 1,  // finished with o.d exact: escaped, or made `limit` updates
    ORBIT_PEND = 2,  // escaped within the round's unchecked block: the dwell is in
                     // (o.d, o.d + K], o keeps the block's starting state
};

// Updates per unchecked block of a perimeter-query round after the short
// first rounds of query_group.  The short rounds take the orbits that escape
// early, so the long ones serve orbits that run long (32 at n = 16384: levels 2
// and 3 at 190 and 387 us against 190 and 371).
constexpr uint32_t kQueryRound = 64;
// Whole perimeters of small regions in a batch (zoomed frames, whose orbits all
// outlive the short rounds): blocks of this size from the first round.
constexpr uint32_t kQueryRoundBatch = 32;
// The CTA-wide query of the paper's SBR / MBR mappings: blocks of 32 from
// the first round.
constexpr uint32_t kQueryRoundCta = 32;

// Advance an orbit by up to K updates (a power of two) without passing
// `limit`.  An orbit still running after a round has made more updates than
// any orbit that finished (or became pending) in it: its dwell is strictly
// larger.  A pending orbit needs orbit_resolve only if its exact dwell is
// wanted.
template <uint32_t K>
__device__ __forceinline__ uint32_t orbit_step(Orbit &o, uint32_t limit)
{
    if (o.d >= limit)
        return ORBIT_DONE;
    if (o.fast && limit - o.d >= K) {
        float x = o.x, y = o.y;
#pragma unroll
        for (uint32_t k = 0; k < K; ++k)
            z_update(x, y, o.cr, o.ci);
        if (!z_bounded(x, y))
            return ORBIT_PEND;
        o.x = x;
        o.y = y;
        o.d += K;
        return o.d >= limit ? ORBIT_DONE : ORBIT_RUN;
    }
    for (uint32_t k = 0; k < K; ++k) {
        if (o.d >= limit || !z_bounded(o.x, o.y))
            return ORBIT_DONE;
        z_update(o.x, o.y, o.cr, o.ci);
        ++o.d;
    }
    // (the last state is tested here as a block's is: an orbit that it ends
    // would be taken for one that outlives those of the same dwell)
    return (o.d >= limit || !z_bounded(o.x, o.y)) ? ORBIT_DONE : ORBIT_RUN;
}

// Exact dwell of an orbit left pending by orbit_step<K>: its starting state
// z_d passed the test and z_{d + K} failed; halving the gap finds the first
// failing state (K - 1 updates, log2(K) tests, no branches that differ by
// lane).
template <uint32_t K>
__device__ __forceinline__ void orbit_resolve(Orbit &o)
{
    float x = o.x, y = o.y;
    uint32_t d = o.d;
#pragma unroll
    for (uint32_t h = K / 2u; h >= 1u; h >>= 1) {
        float tx = x, ty = y;
#pragma unroll
        for (uint32_t k = 0; k < h; ++k)
            z_update(tx, ty, o.cr, o.ci);
        if (z_bounded(tx, ty)) {
            x = tx;
            y = ty;
            d += h;
        }
    }
    o.x = x;
    o.y = y;
    o.d = d + 1u;
}

// Region record of the offset lookup tables (Sec. 5.2): origin and clipped
// extent, 16 bits each (n <= 65536 so x0, y0, w-1, h-1 < 65536).
struct Region {
    uint32_t x0, y0, w, h;
};

__device__ __forceinline__ uint2 pack_region(uint32_t x0, uint32_t y0, uint32_t w, uint32_t h)
{
    return make_uint2(x0 | (y0 << 16), (w - 1u) | ((h - 1u) << 16));
}

__device__ __forceinline__ Region unpack_region(uint2 e)
{
    Region g;
    g.x0 = e.x & 0xffffu;
    g.y0 = e.x >> 16;
    g.w = (e.y & 0xffffu) + 1u;
    g.h = (e.y >> 16) + 1u;
    return g;
}

// Number of perimeter pixels of a w x h region (outermost rows and columns).
__device__ __forceinline__ uint32_t perimeter_size(uint32_t w, uint32_t h)
{
    return (w <= 2u || h <= 2u) ? w * h : 2u * w + 2u * (h - 2u);
}

// k-th perimeter pixel: top row, bottom row, left column, right column
// (columns without the corners), so neighbouring k are neighbouring pixels.
__device__ __forceinline__ void perimeter_pixel(const Region &g, uint32_t k, uint32_t &px,
                                                uint32_t &py)
{
    if (g.w <= 2u || g.h <= 2u) {
        px = g.x0 + k % g.w;
        py = g.y0 + k / g.w;
        return;
    }
    if (k < g.w) {
        px = g.x0 + k;
        py = g.y0;
    } else if (k < 2u * g.w) {
        px = g.x0 + (k - g.w);
        py = g.y0 + g.h - 1u;
    } else {
        const uint32_t j = k - 2u * g.w, hh = g.h - 2u;
        px = (j < hh) ? g.x0 : g.x0 + g.w - 1u;
        py = g.y0 + 1u + ((j < hh) ? j : j - hh);
    }
}

__device__ __forceinline__ bool on_perimeter(const Region &g, uint32_t px, uint32_t py)
{
    return px == g.x0 || py == g.y0 || px == g.x0 + g.w - 1u || py == g.y0 + g.h - 1u;
}

// Cooperative fill of the rectangle g with value v by `nthr` threads
// (thread index `t`).  Each row is cut at 16-byte boundaries of the map; full
// 16-byte chunks take one 128-bit store, the partial chunks at the row ends
// take scalar stores.  The map base must be 16-byte aligned.
__device__ __forceinline__ void fill_rect(uint32_t *__restrict__ map, uint32_t n, const Region &g,
                                          uint32_t v, uint32_t t, uint32_t nthr)
{
    const uint32_t cpr = (g.w + 3u) / 4u + 1u;  // chunks per row, an upper bound for any alignment
    const uint4 v4 = make_uint4(v, v, v, v);
    uint32_t row = t / cpr, c = t - row * cpr;   // then advanced without dividing
    while (row < g.h) {
        const size_t start = (size_t)(g.y0 + row) * n + g.x0;
        const size_t end = start + g.w;
        const size_t e0 = ((start >> 2) + c) << 2;
        if (e0 < end) {
            if (e0 >= start && e0 + 4u <= end) {
                *reinterpret_cast<uint4 *>(map + e0) = v4;
            } else {
#pragma unroll
                for (uint32_t k = 0; k < 4u; ++k)
                    if (e0 + k >= start && e0 + k < end)
                        map[e0 + k] = v;
            }
        }
        c += nthr;
        while (c >= cpr) {
            c -= cpr;
            ++row;
        }
    }
}

// Warp fill of a band of the deferred-fill list.  Rows of at least 128
// pixels go one at a time, the lanes striding over the row's whole 16-byte
// chunks (one 128-bit store, a pointer step and a compare each), with the at
// most 3 + 3 pixels outside them stored singly; narrower bands use fill_rect.
__device__ __forceinline__ void fill_band_warp(uint32_t *__restrict__ map, uint32_t n,
                                               const Region &g, uint32_t v, uint32_t lane)
{
    if (g.w < 128u) {
        fill_rect(map, n, g, v, lane, 32u);
        return;
    }
    const uint4 v4 = make_uint4(v, v, v, v);
    for (uint32_t row = 0; row < g.h; ++row) {
        const size_t start = (size_t)(g.y0 + row) * n + g.x0;
        const size_t end = start + g.w;
        const size_t a4 = (start + 3u) >> 2, b4 = end >> 2;  // whole chunks [a4, b4)
        uint4 *q = reinterpret_cast<uint4 *>(map) + a4 + lane;
        uint4 *const qe = reinterpret_cast<uint4 *>(map) + b4;
        for (; q < qe; q += 32)
            *q = v4;
        if (lane < 3u && start + lane < (a4 << 2))
            map[start + lane] = v;
        if (lane >= 3u && lane < 6u && (b4 << 2) + (lane - 3u) < end)
            map[(b4 << 2) + (lane - 3u)] = v;
    }
}

// ---------------------------------------------------------------------------
// Perimeter uniformity queries for regions that split when not uniform.
//
// Such a region needs only the answer "all perimeter dwells equal, and to
// what", not the dwells themselves (its children evaluate their own
// perimeters).  The orbits of a group of 32 perimeter pixels advance in
// rounds; running orbits stay in lockstep, so as soon as one orbit has
// finished while another still runs, their dwells differ and the query
// stops.  Once one group has finished with a common dwell w, later groups
// stop at w + 1 updates: more updates than w already means a different dwell.
// ---------------------------------------------------------------------------
constexpr unsigned kLaneMask = 0xffffffffu;

// Outcome of query_group.
enum : uint32_t {
    GROUP_SAME = 0,    // every dwell of the group is exact in d (or at least the limit)
    GROUP_DIFFER = 1,  // two dwells of the group differ
    GROUP_STOP = 2,    // another warp found the region non-uniform
};

// Rounds between issuing a load of a region's query state and using it, for
// one frame.  A batch keeps enough warps resident to hide the load, and there
// a late stop costs more than the wait, so it uses the value one round later.
constexpr uint32_t kPollLag = 8;
constexpr uint32_t kNone32 = 0xffffffffu;

// K unchecked updates of NS orbits (one or two, side by side).
template <uint32_t K, int NS>
__device__ __forceinline__ void run_block(float *x, float *y, const float *cr, const float *ci)
{
    if (NS == 1) {
#pragma unroll
        for (uint32_t k = 0; k < K; ++k)
            z_update(x[0], y[0], cr[0], ci[0]);
    } else {
        f32x2 X = pack2(x[0], x[NS - 1]), Y = pack2(y[0], y[NS - 1]);
        const f32x2 CR = pack2(cr[0], cr[NS - 1]), CI = pack2(ci[0], ci[NS - 1]);
#pragma unroll
        for (uint32_t k = 0; k < K; ++k)
            z_update2(X, Y, CR, CI);
        unpack2(X, x[0], x[NS - 1]);
        unpack2(Y, y[0], y[NS - 1]);
    }
}

// Exact dwells of orbits whose state (x, y) at count d passed the test and
// whose state K updates later failed (pend): halving the gap finds the first
// failing state (K - 1 updates, log2(K) tests, the same on every lane).  The
// search stops, and returns true, at the first half that some of these orbits
// pass and others do not: their dwells differ.
template <uint32_t K, int NS>
__device__ __forceinline__ bool resolve_block(const float *x0, const float *y0, const float *cr,
                                              const float *ci, const bool *pend, uint32_t base,
                                              uint32_t *d)
{
    static_assert(K <= 64u && (K & (K - 1u)) == 0u, "blocks of up to 64 updates, a power of two");
    float x[NS], y[NS];
    uint32_t r[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        x[i] = x0[i];
        y[i] = y0[i];
        r[i] = base;
    }
#pragma unroll
    for (uint32_t h = K / 2u; h >= 1u; h >>= 1) {
        float tx[NS], ty[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            tx[i] = x[i];
            ty[i] = y[i];
        }
        // (an unrolled run_block of h updates)
        if (h >= 32u)
            run_block<32u, NS>(tx, ty, cr, ci);
        else if (h == 16u)
            run_block<16u, NS>(tx, ty, cr, ci);
        else if (h == 8u)
            run_block<8u, NS>(tx, ty, cr, ci);
        else if (h == 4u)
            run_block<4u, NS>(tx, ty, cr, ci);
        else if (h == 2u)
            run_block<2u, NS>(tx, ty, cr, ci);
        else
            run_block<1u, NS>(tx, ty, cr, ci);
        bool passed = false, failed = false;
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const bool ok = z_bounded(tx[i], ty[i]);
            passed = passed || (pend[i] && ok);
            failed = failed || (pend[i] && !ok);
            if (ok) {
                x[i] = tx[i];
                y[i] = ty[i];
                r[i] += h;
            }
        }
        if (__any_sync(kLaneMask, passed) && __any_sync(kLaneMask, failed))
            return true;
    }
#pragma unroll
    for (int i = 0; i < NS; ++i)
        if (pend[i])
            d[i] = r[i] + 1u;
    return false;
}

// The orbits of up to 32 * NS perimeter pixels (NS a lane, `active`) advance
// in lockstep rounds of unchecked blocks: 8, 8, 16, then K updates (rnd = 3
// skips the short ones).  Most perimeter orbits outside the set escape within
// a few updates, and a short first block and the short search after it cost
// them about 15 updates where a K-update block and its search cost 2K - 1.
// The rounds end as soon as an orbit escapes: if another still runs, or never
// will escape, two dwells differ; else all escaped in this round and their
// dwells are resolved.  PROVE: an orbit is proven to stay (its dwell is max_dwell)
// when it enters its capture disc or repeats the state it had at rounds 1, 2,
// 4, 8, ... of the long ones, so a cycle is seen within twice the rounds it
// took to enter it.  w: the region's common dwell as far as known (kNone32:
// none yet); orbits stop at w + 1.  ps (or NULL): the region's shared state
// {common dwell, differs}, read along the way, `lag` rounds between a load and
// its use.  On GROUP_SAME d holds the dwells (above w: anything above w).  `it`
// gains the updates that proofs spared.
template <uint32_t K, int NS, bool PROVE>
__device__ __forceinline__ uint32_t query_group(const PixelMap &pm, uint32_t max_dwell,
                                                const uint32_t *px, const uint32_t *py,
                                                const bool *active, uint32_t rnd, uint32_t w,
                                                const volatile uint32_t *ps, uint32_t lag,
                                                uint32_t lane, uint32_t *d, Updates &it)
{
    float x[NS], y[NS], cr[NS], ci[NS];
    float bx[NS], by[NS], ax[NS], ay[NS], r2[NS];
    bool run[NS], pend[NS], may[NS];
    bool plain = false;
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const float2 c = pixel_c(pm, px[i], py[i]);
        cr[i] = c.x;
        ci[i] = c.y;
        x[i] = y[i] = 0.0f;
        bx[i] = by[i] = ax[i] = ay[i] = 0.0f;
        r2[i] = -1.0f;
        run[i] = active[i];
        pend[i] = false;
        may[i] = may_capture(c.x, c.y);
        d[i] = 0;
        plain = plain || (active[i] && !escape_absorbing(c.x, c.y));
    }
    uint32_t limit = (w != kNone32) ? min(max_dwell, w + 1u) : max_dwell;
    if (__any_sync(kLaneMask, plain)) {
        // points with |c| near 2 or above (most escape at once): tested updates
        // for the whole group, from z = 0, to 8 of them, then 32, 128, ...;
        // orbits that ended and orbits that reached the length differ.  Each
        // orbit run to its own end instead: level 0 of (-2.5, -0.5, -1, 1), g = 1,
        // n = 512, at caps 2048 / 8192 / 65536 66 / 229 / 1758 us, this way 13 / 13 /
        // 12.  (Lockstep rounds as below in a function of their own cost the other
        // queries of its callers registers: n = 65536 9.90 -> 10.0 ms.)
        for (uint32_t len = min(limit, 8u);; len = len > limit / 4u ? limit : 4u * len) {
            uint32_t nx = w, ny = 0;
            if (ps != nullptr && lane == 0) {
                nx = ps[0];
                ny = ps[1];
            }
            bool ended = false, reached = false;
#pragma unroll
            for (int i = 0; i < NS; ++i)
                if (active[i]) {
                    d[i] = dwell_tested(cr[i], ci[i], len);
                    ended = ended || d[i] < len;
                    reached = reached || d[i] >= len;
                }
            if (len >= limit || !__any_sync(kLaneMask, reached))
                return GROUP_SAME;
            if (__any_sync(kLaneMask, ended))
                return GROUP_DIFFER;
            if (ps != nullptr) {
                w = __shfl_sync(kLaneMask, nx, 0);
                if (__shfl_sync(kLaneMask, ny, 0))
                    return GROUP_STOP;
                limit = (w != kNone32) ? min(max_dwell, w + 1u) : max_dwell;
            }
        }
    }
    uint32_t n = 0;  // updates made by the running orbits
    uint32_t nx = w, ny = 0, age = 0, step;
    for (;; ++rnd) {
        if (ps != nullptr && age == 0 && lane == 0) {
            nx = ps[0];
            ny = ps[1];
        }
        step = rnd < 2u ? 8u : rnd == 2u ? 16u : K;
        if (n + step > limit || n + step < n) {
            // less than a block left: tested updates (none if w fell below n)
            for (; n < limit; ++n)
#pragma unroll
                for (int i = 0; i < NS; ++i)
                    if (run[i]) {
                        run[i] = z_bounded(x[i], y[i]);
                        d[i] = n;
                        z_update(x[i], y[i], cr[i], ci[i]);
                    }
#pragma unroll
            for (int i = 0; i < NS; ++i)
                if (run[i])
                    d[i] = n;
            return GROUP_SAME;
        }
        if (PROVE && rnd >= 3u && ((rnd - 3u) & (rnd - 4u)) == 0u) {
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                bx[i] = x[i];
                by[i] = y[i];
                if (run[i] && may[i])
                    capture_disc(cr[i], ci[i], x[i], y[i], ax[i], ay[i], r2[i]);
            }
        }
        float tx[NS], ty[NS];
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            tx[i] = x[i];
            ty[i] = y[i];
        }
        if (rnd < 2u)
            run_block<8u, NS>(tx, ty, cr, ci);
        else if (rnd == 2u)
            run_block<16u, NS>(tx, ty, cr, ci);
        else
            run_block<K, NS>(tx, ty, cr, ci);
        n += step;
        bool any_run = false, any_pend = false;
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const bool ok = z_bounded(tx[i], ty[i]);
            pend[i] = run[i] && !ok;
            if (ok) {
                x[i] = tx[i];
                y[i] = ty[i];
            }
            const float ux = x[i] - ax[i], uy = y[i] - ay[i];
            const bool in = PROVE && rnd >= 3u && (__fmaf_rn(ux, ux, __fmul_rn(uy, uy)) < r2[i] ||
                                          (x[i] == bx[i] && y[i] == by[i]));
            if (run[i] && ok)
                d[i] = in ? max_dwell : n;
            if (run[i] && ok && in)
                it.spared += max_dwell - n;
            // (at the limit an orbit has ended: its dwell may equal that of
            // one whose last state escaped)
            run[i] = run[i] && ok && !in && n < limit;
            any_run = any_run || run[i];
            any_pend = any_pend || pend[i];
        }
        any_run = __any_sync(kLaneMask, any_run);
        any_pend = __any_sync(kLaneMask, any_pend);
        if (any_pend)
            break;
        if (!any_run)
            return GROUP_SAME;
        if (ps != nullptr && ++age == lag) {
            age = 0;
            w = __shfl_sync(kLaneMask, nx, 0);
            if (__shfl_sync(kLaneMask, ny, 0))
                return GROUP_STOP;
            limit = (w != kNone32) ? min(max_dwell, w + 1u) : max_dwell;
        }
    }
    bool left = false;
#pragma unroll
    for (int i = 0; i < NS; ++i)
        left = left || run[i];
    if (__any_sync(kLaneMask, left))
        return GROUP_DIFFER;
    bool differ;
    if (step == 8u)
        differ = resolve_block<8u, NS>(x, y, cr, ci, pend, n - step, d);
    else if (step == 16u)
        differ = resolve_block<16u, NS>(x, y, cr, ci, pend, n - step, d);
    else
        differ = resolve_block<K, NS>(x, y, cr, ci, pend, n - step, d);
    return differ ? GROUP_DIFFER : GROUP_SAME;
}

// The dwells of a group (NS a lane): their least and greatest.
template <int NS>
__device__ __forceinline__ void group_range(const bool *active, const uint32_t *d, uint32_t &vmin,
                                            uint32_t &vmax)
{
    vmin = kNone32;
    vmax = 0u;
#pragma unroll
    for (int i = 0; i < NS; ++i)
        if (active[i]) {
            vmin = min(vmin, d[i]);
            vmax = max(vmax, d[i]);
        }
    vmin = __reduce_min_sync(kLaneMask, vmin);
    vmax = __reduce_max_sync(kLaneMask, vmax);
}

// A group of up to 32 * NS of the perimeter pixels of g (P pixels), a stride
// apart: pixels first + k * stride, k = base, base + 1, ...
template <uint32_t K, int NS, bool PROVE>
__device__ __forceinline__ uint32_t spread_group(const PixelMap &pm, uint32_t max_dwell, const Region &g,
                                                 uint32_t first, uint32_t stride, uint32_t base,
                                                 uint32_t P, uint32_t rnd, uint32_t w,
                                                 const volatile uint32_t *ps, uint32_t lag, uint32_t lane,
                                                 uint32_t &vmin, uint32_t &vmax, Updates &it)
{
    uint32_t px[NS], py[NS], d[NS];
    bool active[NS];
#pragma unroll
    for (int i = 0; i < NS; ++i) {
        const uint32_t k = first + (base + lane + 32u * (uint32_t)i) * stride;
        active[i] = k < P;
        px[i] = g.x0;
        py[i] = g.y0;
        if (active[i])
            perimeter_pixel(g, k, px[i], py[i]);
    }
    const uint32_t r = query_group<K, NS, PROVE>(pm, max_dwell, px, py, active, rnd, w, ps, lag, lane, d, it);
#pragma unroll
    for (int i = 0; i < NS; ++i)
        if (active[i])
            it += d[i];
    if (r == GROUP_SAME)
        group_range<NS>(active, d, vmin, vmax);
    return r;
}

// One warp queries the whole perimeter of g, NS orbits a lane.  Returns true
// and the common dwell in *w_out if the perimeter is uniform; `it` gains the
// updates made.
template <uint32_t K, int NS, bool PROVE>
__device__ __forceinline__ bool warp_perimeter_uniform(const PixelMap &pm, uint32_t max_dwell,
                                                       const Region &g, uint32_t lane, uint32_t rnd,
                                                       uint32_t *w_out, Updates &it)
{
    const uint32_t P = perimeter_size(g.w, g.h);
    const uint32_t groups = (P + 32u * NS - 1u) / (32u * NS);
    uint32_t w = kNone32, vmin = 0, vmax = 0;
    for (uint32_t j = 0; j < groups; ++j) {
        const uint32_t r = spread_group<K, NS, PROVE>(pm, max_dwell, g, j, groups, 0u, P, rnd, w, nullptr, 0u, lane,
                                               vmin, vmax, it);
        if (r != GROUP_SAME || vmin != vmax || (w != kNone32 && vmin != w))
            return false;
        w = vmin;
    }
    *w_out = w;
    return true;
}

// All warps of a CTA query the perimeter of g together; warps share the
// verdict through s_flag (1 = not uniform) and the common dwell through s_w
// (0xffffffff = none yet).  The caller sets *s_flag = 0 and *s_w = 0xffffffff
// and synchronises the CTA before the call; the call ends with a CTA barrier.
__device__ __forceinline__ bool cta_perimeter_uniform(const PixelMap &pm, uint32_t max_dwell,
                                                      const Region &g, uint32_t tid, uint32_t T,
                                                      uint32_t *s_flag, uint32_t *s_w,
                                                      uint32_t *w_out, Updates &it)
{
    const uint32_t P = perimeter_size(g.w, g.h);
    const uint32_t lane = tid & 31u;
    volatile uint32_t *vflag = s_flag;
    volatile uint32_t *vw = s_w;
    for (uint32_t base = (tid & ~31u); base < P; base += T) {
        if (__shfl_sync(kLaneMask, *vflag, 0))
            break;
        const uint32_t k = base + lane;
        const bool active = k < P;
        const unsigned amask = __ballot_sync(kLaneMask, active);
        uint32_t px = g.x0, py = g.y0;
        if (active)
            perimeter_pixel(g, k, px, py);
        Orbit o = orbit_start(pixel_c(pm, px, py));
        uint32_t stt = active ? ORBIT_RUN : ORBIT_DONE;
        bool differ = false, stop = false;
        for (;;) {
            // one value per warp, so every lane uses the same limit
            const uint32_t wv = __shfl_sync(kLaneMask, *vw, 0);
            const uint32_t limit = (wv != 0xffffffffu) ? min(max_dwell, wv + 1u) : max_dwell;
            if (stt == ORBIT_RUN)
                stt = orbit_step<kQueryRoundCta>(o, limit);
            const unsigned dm = __ballot_sync(kLaneMask, stt != ORBIT_RUN) & amask;
            if (dm == amask)
                break;
            if (dm) {
                differ = true;
                break;
            }
            if (__shfl_sync(kLaneMask, *vflag, 0)) {
                stop = true;
                break;
            }
        }
        if (!stop && !differ && stt == ORBIT_PEND)
            orbit_resolve<kQueryRoundCta>(o);
        if (active)
            it += o.d;
        if (stop)
            break;
        if (differ) {
            if (lane == 0)
                *vflag = 1u;
            break;
        }
        const uint32_t vmin = __reduce_min_sync(kLaneMask, active ? o.d : 0xffffffffu);
        const uint32_t vmax = __reduce_max_sync(kLaneMask, active ? o.d : 0u);
        if (lane == 0) {
            if (vmin != vmax) {
                *vflag = 1u;
            } else {
                const uint32_t old = atomicCAS(s_w, 0xffffffffu, vmin);
                if (old != 0xffffffffu && old != vmin)
                    *vflag = 1u;
            }
        }
        __syncwarp();
    }
    __syncthreads();
    const bool uniform = (*vflag == 0u);
    *w_out = *vw;
    __syncthreads();
    return uniform;
}

__device__ __forceinline__ uint32_t ceil_div_u32(uint32_t a, uint32_t b)
{
    return a / b + (a % b != 0u);
}

// Number of non-empty children of a region (r x r split into side sc,
// clipped to the region).
__device__ __forceinline__ uint32_t child_count(const Region &g, uint32_t sc, uint32_t r)
{
    const uint32_t cx = min(r, ceil_div_u32(g.w, sc));
    const uint32_t cy = min(r, ceil_div_u32(g.h, sc));
    return cx * cy;
}

// j-th non-empty child (row-major over the cx x cy children).
__device__ __forceinline__ uint2 child_region(const Region &g, uint32_t sc, uint32_t r, uint32_t j)
{
    const uint32_t cx = min(r, ceil_div_u32(g.w, sc));
    const uint32_t a = j % cx, b = j / cx;
    const uint32_t x = g.x0 + a * sc, y = g.y0 + b * sc;
    const uint32_t w = min(sc, g.x0 + g.w - x), h = min(sc, g.y0 + g.h - y);
    return pack_region(x, y, w, h);
}

}  // namespace ask
