// vicp_search.cuh -- device code of the NNS (Alg. 4) shared by the
// single-grid kernels and the batched iteration kernel: the scan of a root
// voxel's CSR segment, and the exact global search over the brick levels.
#pragma once

#include "vicp_device.cuh"

namespace vicp {

// A root segment longer than this is scanned by a group of lanes, not by the
// query's own thread (a warp waits for its longest segment).  On the 226k
// scene 48 leaves 9-18k of the 226k queries to such groups (32: 27-38k)
// while the longest light segment of a warp grows by a sixth: measured step
// 107.5 -> 105.9 us.
constexpr unsigned HEAVY = 48;

// Nearest point of the CSR run [a, b) to s by one thread: 16-byte loads of
// (x, y, z, index), eight in flight, then four, then the last three at once
// with the index held at the run's last point (a point examined twice changes
// no minimum), so that a short run is one round of loads and not one round
// trip a point.  Returns the smaller of `best` and the run's (distance bits,
// index) key; ~0 when both are empty.
__device__ __forceinline__ unsigned long long segment_min(const float4 *__restrict__ csr, unsigned a, unsigned b,
                                                          float3 s, unsigned long long best = ~0ull)
{
    unsigned k = a;
    for (; k + 8 <= b; k += 8) {
        float4 q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            q[u] = __ldg(csr + k + u);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            best = umin64(best, nn_key(dist2(s, q[u]), __float_as_int(q[u].w)));
    }
    if (k + 4 <= b) {
        float4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            q[u] = __ldg(csr + k + u);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            best = umin64(best, nn_key(dist2(s, q[u]), __float_as_int(q[u].w)));
        k += 4;
    }
    if (k < b) {
        float4 q[3];
#pragma unroll
        for (int u = 0; u < 3; ++u)
            q[u] = __ldg(csr + min(k + u, b - 1u));
#pragma unroll
        for (int u = 0; u < 3; ++u)
            best = umin64(best, nn_key(dist2(s, q[u]), __float_as_int(q[u].w)));
    }
    return best;
}

// ---------------------------------------------------------------------------
// Near global queries.  Most points that take the global search lie just
// outside the grid (the grid is the target's bounding box, so a flat side of
// the target lies on its face and noise alone puts half of the matching
// points outside): on the scenes and objects measured, 60-99% of them, half
// of those within three voxels of their nearest point.  For them the grid
// itself bounds the answer: the voxel nearest to the point has a root label,
// and any point of that root's segment is at a distance D the nearest point
// cannot exceed.  The localised search reads that segment anyway (the same
// loads as for a point inside), so it leaves the seed (D, index) in the
// query's own nn / d2 entries, and where the voxels that can hold a point
// within D are few rows, the query is listed as near.  A group of 1 to 32
// lanes then takes those rows (all voxels of one y and z, at most 32 along
// x), a row a lane, the rows nearest to the query first: one window of
// occupancy bits, and the occupied voxels of the window are one run of the
// CSR store.  There is no chain from box to box as in the brick search
// below, and many queries share a warp.  (Where a voxel holds many points
// the rows would hold hundreds, and the brick search, which narrows D brick
// by brick, is the better one.  On 256 pairs of objects, 14.7% of whose
// queries are global, a batch of 40 iterations went from 47.5 to 25.2 ms;
// NEAR_WORK 96: 27.7, 512: 24.5, but the 226k scene's registration 2% longer.)
//
// Exactness.  A point p with computed squared distance <= D2 is, in exact
// arithmetic, within sqrt(D2) (1 + 2^-22) of s (rounding is monotone; below
// 1e-18 a difference's square underflows, hence the floor at 1e-36).  Rows
// and window ends are those of the ball of that radius in voxel units,
// widened by a margin that covers the rounding of scaled coordinates (three
// operations, 2^-24 of their size each, where the margin takes 1e-6 of it).
// Every candidate's distance is computed as everywhere else, so the
// (distance, index) minimum is that of a scan of all target points.
// ---------------------------------------------------------------------------
constexpr int NEAR_SHIFT_MIN = 0;     // a near query gets one lane at least
constexpr int HEAVY_SHIFT_MIN = 2;    // a dense segment four
constexpr float NEAR_R2 = 15.9f;      // squared distance of the seed in voxels, at most: beyond it the brick search
constexpr int NEAR_WORK = 256;        // ... which also takes what has more rows times points a voxel than this
constexpr int NEAR_SEED = 16;         // points of a root segment examined for the seed
constexpr int NEAR_OUTSIDE_MAX = 64;  // with more target points outside the grid: the brick search

// Whether a query s with a seed at squared distance d2, from a root segment
// of `dense` points, is near: at most 3 voxels, so at most 8 voxels along
// every axis, and few points expected ((2r + 1)^2 <= 8 r^2 + 2 rows of
// `dense`).  A coordinate of 2^20 voxels and more has too few bits for that
// count of voxels.
__device__ __forceinline__ bool near_seed(float3 s, float d2, float inv_h, unsigned dense)
{
    const float r2 = d2 * (inv_h * inv_h);   // (not a number, or infinite: far)
    return r2 <= NEAR_R2 && (8.0f * r2 + 2.0f) * (float)dense <= (float)NEAR_WORK &&
           fmaxf(fmaxf(fabsf(s.x), fabsf(s.y)), fabsf(s.z)) * inv_h <= 1048576.0f;
}

// Square root to 2^-22 (what it is used for has a margin of 1e-3 voxels).
__device__ __forceinline__ float near_sqrt(float x)
{
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

struct NearBox {
    int x0, x1, y0, y1, z0, z1;   // voxels, inclusive
};

__device__ __forceinline__ int near_voxel(float c, float o, float inv_h, int n)
{
    const float f = __fmul_rn(__fsub_rn(c, o), inv_h);
    return min((int)fminf(fmaxf(f, 0.0f), 2147483520.0f), n - 1);
}

// The grid voxel nearest to s (its own voxel when s lies inside); `inside`
// as voxel_coords.  -1 for a point with a non-finite coordinate.
__device__ __forceinline__ int nearest_voxel(const GridGeom &g, float3 s, bool &inside)
{
    int ix, iy, iz;
    inside = voxel_coords(g, s.x, s.y, s.z, ix, iy, iz);
    if (!inside) {
        if (!(isfinite(s.x) && isfinite(s.y) && isfinite(s.z)))
            return -1;
        ix = near_voxel(s.x, g.ox, g.inv_h, g.nx);
        iy = near_voxel(s.y, g.oy, g.inv_h, g.ny);
        iz = near_voxel(s.z, g.oz, g.inv_h, g.nz);
    }
    return ix + g.nx * (iy + g.ny * iz);
}

// Lanes each of n near queries or dense segments gets, as a power of two: as
// many as `lanes` resident lanes allow, 2^least to 32 (few queries: one short
// round trip each; many: several to a warp, whose chains of loads overlap).
__device__ __forceinline__ int group_shift(int n, int lanes, int least)
{
    if (n <= 0 || n <= lanes >> 5)
        return 5;
    return max(least, 31 - __clz(max(lanes / n, 1)));
}

// Warp minimum of (distance bits, index) keys: the smallest distance, then
// the smallest index at it -- two single-instruction warp reductions.
__device__ __forceinline__ unsigned long long warp_min_key(unsigned long long v)
{
    const unsigned d = __reduce_min_sync(FULL_MASK, (unsigned)(v >> 32));
    const unsigned i = __reduce_min_sync(FULL_MASK, (unsigned)(v >> 32) == d ? (unsigned)v : 0xffffffffu);
    return ((unsigned long long)d << 32) | i;
}

// Minimum key over each aligned group of G lanes (the whole warp calls it).
__device__ __forceinline__ unsigned long long group_min(unsigned long long v, int G)
{
    if (G == 32)
        return warp_min_key(v);
    for (int o = G / 2; o > 0; o >>= 1)
        v = umin64(v, __shfl_xor_sync(FULL_MASK, v, o));
    return v;
}

// The points of occupied voxels (bits, at `key` on) of a row as runs of the
// store: next() takes some of the bits and gives their run.  In the CSR store
// a row is one run, from the first occupied voxel's offset to the one past
// the last's (both of which the build writes).
struct CsrRows {
    const unsigned *occ, *off;
    unsigned cap;
    const float4 *csr;
    __device__ __forceinline__ void next(int key, unsigned &bits, unsigned &a, unsigned &e) const
    {
        a = __ldg(off + key + (__ffs(bits) - 1));
        e = min(__ldg(off + key + (32 - __clz(bits))), cap);
        bits = 0u;
    }
};

// On the sparse grid, whose segments lie in slot order: a lookup and a run
// an occupied voxel.
struct HashedRows {
    const unsigned *occ, *off;
    unsigned cap;
    const float4 *csr;
    const unsigned *okeys;
    unsigned omask;
    int oshift;
    __device__ __forceinline__ void next(int key, unsigned &bits, unsigned &a, unsigned &e) const
    {
        const int slot = hash_find(okeys, omask, oshift, (unsigned)(key + __ffs(bits) - 1));
        bits &= bits - 1u;
        a = e = 0u;
        if (slot >= 0) {
            a = __ldg(off + slot);
            e = min(__ldg(off + slot + 1), cap);
        }
    }
};

// The runs [a, a + c) of the lanes of each aligned group of G lanes, scanned
// by the group.  Runs of at most RUN_OWN points are scanned by their own
// lanes; where a run of the warp is longer (a dense voxel holds hundreds of
// points, and one lane would keep the others waiting) the groups deal all
// points of their runs out over their lanes: point t of the concatenated
// runs belongs to the first lane whose inclusive count exceeds t, found by
// bisection over the lanes.
constexpr unsigned RUN_OWN = 8;

__device__ __forceinline__ unsigned long long scan_runs(const float4 *__restrict__ csr, unsigned a, unsigned c,
                                                        float3 s, unsigned long long best, int sub, int G)
{
    if (G == 1 || !__any_sync(FULL_MASK, c > RUN_OWN))
        return c ? segment_min(csr, a, a + c, s, best) : best;
    unsigned incl = c;
    for (int d = 1; d < G; d <<= 1) {
        const unsigned y = __shfl_up_sync(FULL_MASK, incl, d, G);
        if (sub >= d)
            incl += y;
    }
    const unsigned total = __shfl_sync(FULL_MASK, incl, G - 1, G);
    const unsigned base = a + c - incl;   // point t of the group is point base + t of the store
    const unsigned most = __reduce_max_sync(FULL_MASK, total);
    for (unsigned t0 = 0u; t0 < most; t0 += 4u * G) {
        float4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const unsigned t = t0 + (unsigned)(u * G + sub);
            int own = 0;
            for (int step = G >> 1; step > 0; step >>= 1)
                if (__shfl_sync(FULL_MASK, incl, own + step - 1, G) <= t)
                    own += step;
            const unsigned p = __shfl_sync(FULL_MASK, base, own, G) + t;
            q[u].w = 0.0f;
            if (t < total)
                q[u] = __ldg(csr + p);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (t0 + (unsigned)(u * G + sub) < total)
                best = umin64(best, nn_key(dist2(s, q[u]), __float_as_int(q[u].w)));
    }
    return best;
}

// The k-th index of [a, b] in the order of distance from c (a <= c <= b).
__device__ __forceinline__ int outward(int k, int a, int b, int c)
{
    const int t = min(c - a, b - c);
    if (k <= 2 * t)
        return c + ((k & 1) ? (k + 1) / 2 : -(k / 2));
    return c - a > b - c ? c - (k - t) : c + (k - t);
}

// One near query by an aligned group of G lanes (lane `sub` of them), from
// the seed `best` on; on = false: a group without a query.  The whole warp
// calls it.  Returns the group's minimum on each of its lanes.  The next
// row's occupancy words are loaded while a row is scanned, and the best
// distance is shared after every round of G rows.
template <class Rows>
__device__ __forceinline__ unsigned long long near_search(const GridGeom &g, const Rows &rows, float3 s,
                                                          unsigned long long best, bool on, int sub, int G,
                                                          unsigned &examined)
{
    const float sx = __fmul_rn(__fsub_rn(s.x, g.ox), g.inv_h), sy = __fmul_rn(__fsub_rn(s.y, g.oy), g.inv_h),
                sz = __fmul_rn(__fsub_rn(s.z, g.oz), g.inv_h);
    const float m = 1e-3f + 1e-6f * (fmaxf(fmaxf(fabsf(sx), fabsf(sy)), fabsf(sz)) +
                                     (float)max(max(g.nx, g.ny), g.nz));
    const float scale = 1.0002f * g.inv_h * g.inv_h;
    const float r2s = fmaxf(__uint_as_float((unsigned)(best >> 32)), 1e-36f) * scale;
    NearBox b{0, 0, 0, 0, 0, 0};
    int ny = 1, n = 0;
    if (on && r2s <= 1.001f * NEAR_R2) {   // (any other seed would be a stale entry)
        const float r = near_sqrt(r2s) + m;
        b.x0 = max((int)floorf(sx - r), 0);
        b.x1 = min((int)floorf(sx + r), g.nx - 1);
        b.y0 = max((int)floorf(sy - r), 0);
        b.y1 = min((int)floorf(sy + r), g.ny - 1);
        b.z0 = max((int)floorf(sz - r), 0);
        b.z1 = min((int)floorf(sz + r), g.nz - 1);
        ny = b.y1 - b.y0 + 1;
        n = b.x0 <= b.x1 && ny > 0 && b.z0 <= b.z1 ? ny * (b.z1 - b.z0 + 1) : 0;
    }
    const int yc = min(max((int)floorf(sy), b.y0), b.y1), zc = min(max((int)floorf(sz), b.z0), b.z1);
    const float inv_ny = __fdividef(1.0f, (float)ny);   // (rows of at most 10 x 10: (row + 1/2) / ny is never near an integer)
    auto locate = [&](int row, int &iy, int &iz) {
        const int kz = (int)(((float)row + 0.5f) * inv_ny);
        iy = outward(row - kz * ny, b.y0, b.y1, yc);
        iz = outward(kz, b.z0, b.z1, zc);
        return b.x0 + g.nx * (iy + g.ny * iz);
    };
    int row = sub, iy = 0, iz = 0, key = 0;
    unsigned lo = 0u, hi = 0u;
    if (row < n) {
        key = locate(row, iy, iz);
        lo = __ldg(rows.occ + (key >> 5));
        hi = __ldg(rows.occ + (key >> 5) + 1);   // (the bits have two words past the last voxel's)
    }
    const int rounds = __reduce_max_sync(FULL_MASK, (n + G - 1) / G);
    for (int r = 0; r < rounds; ++r, row += G) {
        const int jy = iy, jz = iz, jkey = key;
        const unsigned window = __funnelshift_r(lo, hi, jkey & 31);
        if (row + G < n) {
            key = locate(row + G, iy, iz);
            lo = __ldg(rows.occ + (key >> 5));
            hi = __ldg(rows.occ + (key >> 5) + 1);
        }
        unsigned bits = 0u;
        if (row < n && window) {
            const float fy = (float)jy, fz = (float)jz;
            const float gy = fmaxf(fmaxf(fy - sy, sy - (fy + 1.0f)) - m, 0.0f);
            const float gz = fmaxf(fmaxf(fz - sz, sz - (fz + 1.0f)) - m, 0.0f);
            const float r2 = fmaxf(__uint_as_float((unsigned)(best >> 32)), 1e-36f) * scale;
            const float t = r2 - gy * gy - gz * gz;
            if (t >= 0.0f) {
                const float w = near_sqrt(t) + m;
                const int xa = max(b.x0, (int)floorf(sx - w)) - b.x0, xb = min(b.x1, (int)floorf(sx + w)) - b.x0;
                if (xa <= xb)
                    bits = window & (0xffffffffu << xa) & (0xffffffffu >> (31 - xb));
            }
        }
        if (!__any_sync(FULL_MASK, bits != 0u))
            continue;
        do {
            unsigned a = 0u, e = 0u;
            if (bits)
                rows.next(jkey, bits, a, e);
            const unsigned c = e > a ? e - a : 0u;
            examined += c;
            best = scan_runs(rows.csr, a, c, s, best, sub, G);
        } while (__any_sync(FULL_MASK, bits != 0u));
        best = group_min(best, G);
    }
    return best;
}

// ---------------------------------------------------------------------------
// Global search ("Globalsearch" of Alg. 4): the exact nearest target point,
// found without scanning every point.
//
// The grid build groups the stored target points per non-empty 8x8x8 brick
// (contiguous runs of (x, y, z, index)) with each brick's exact float
// bounding box, and groups the bricks per 4x4x4-brick super-brick (a
// contiguous range of brick slots) with the union of their boxes.  For a
// query s, the box bound lb = ((ex*ex + ey*ey) + ez*ez), with e the rounded
// gap between s and the box on each axis, is never larger than the computed
// squared distance from s to any point in the box: rounding is monotone, so
// every operation of the bound is <= the same operation of the distance
// formula.  A warp per query
//   (1) takes the super-brick of smallest bound, and in it the brick of
//       smallest bound, and scans that brick's points (lanes split the run),
//       which gives a first best distance D;
//   (2) visits every super-brick whose bound is <= D, and in it scans each
//       brick whose bound is still <= D, tightening D as it goes;
//   (3) scans the target points that lie outside the grid.
// The result is the same (distance, index) minimum as a scan of all target
// points.  A query with a non-finite coordinate scans all target points.
// ---------------------------------------------------------------------------

// The gap on an axis is max(lo - s, s - hi, 0): at most one difference is
// positive, and rounding keeps each difference's sign.
__device__ __forceinline__ float box_lb2(float3 s, float4 lo, float4 hi)
{
    const float ex = fmaxf(fmaxf(__fsub_rn(lo.x, s.x), __fsub_rn(s.x, hi.x)), 0.0f);
    const float ey = fmaxf(fmaxf(__fsub_rn(lo.y, s.y), __fsub_rn(s.y, hi.y)), 0.0f);
    const float ez = fmaxf(fmaxf(__fsub_rn(lo.z, s.z), __fsub_rn(s.z, hi.z)), 0.0f);
    return __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
}

// Record index of the smallest bound over the warp (lane values lb, k; any
// lane holding the minimum may win: the choice only orders the search).
__device__ __forceinline__ int warp_argmin(unsigned lb, int k)
{
    const unsigned mn = __reduce_min_sync(FULL_MASK, lb);
    return __shfl_sync(FULL_MASK, k, __ffs(__ballot_sync(FULL_MASK, lb == mn)) - 1);
}

// Bound of box record k (as order-preserving bits), and its index range
// [a, b) (the boxes carry their ranges in the w fields).
__device__ __forceinline__ unsigned box_bound(const float4 *__restrict__ box, int k, float3 s)
{
    return __float_as_uint(box_lb2(s, __ldg(box + 2 * k), __ldg(box + 2 * k + 1)));
}

__device__ __forceinline__ uint2 box_range(const float4 *__restrict__ box, int k)
{
    return make_uint2(__float_as_uint(__ldg(box + 2 * k).w), __float_as_uint(__ldg(box + 2 * k + 1).w));
}

// Bound and index range of box record k.
__device__ __forceinline__ void load_rec(const float4 *__restrict__ box, int k, float3 s, unsigned &lb, unsigned &a,
                                         unsigned &b)
{
    const float4 lo = __ldg(box + 2 * k), hi = __ldg(box + 2 * k + 1);
    lb = __float_as_uint(box_lb2(s, lo, hi));
    a = __float_as_uint(lo.w);
    b = __float_as_uint(hi.w);
}

// All lanes scan the run [a, b) of brick-ordered points (four loads in
// flight per lane); returns the warp-wide minimum key (every lane gets it).
__device__ __forceinline__ unsigned long long scan_run(const float4 *__restrict__ bpts, unsigned a, unsigned b,
                                                       float3 s, int lane, unsigned long long best,
                                                       unsigned long long &examined)
{
    unsigned i = a + lane;
    for (; i + 96 < b; i += 128) {
        const float4 q0 = __ldg(bpts + i), q1 = __ldg(bpts + i + 32);
        const float4 q2 = __ldg(bpts + i + 64), q3 = __ldg(bpts + i + 96);
        best = umin64(best, nn_key(dist2(s, q0), __float_as_int(q0.w)));
        best = umin64(best, nn_key(dist2(s, q1), __float_as_int(q1.w)));
        best = umin64(best, nn_key(dist2(s, q2), __float_as_int(q2.w)));
        best = umin64(best, nn_key(dist2(s, q3), __float_as_int(q3.w)));
    }
    for (; i < b; i += 32) {
        const float4 q = __ldg(bpts + i);
        best = umin64(best, nn_key(dist2(s, q), __float_as_int(q.w)));
    }
    examined += b - a;
    return warp_min_key(best);
}

// Scan, in ascending lane order, the bricks of one 32-record chunk whose bound
// (lb, per lane) is <= the current best distance; (ra, rb) are the bricks'
// point ranges.
__device__ __forceinline__ unsigned long long scan_chunk(const float4 *__restrict__ bpts, unsigned lb, unsigned ra,
                                                         unsigned rb, float3 s, int lane, unsigned long long best,
                                                         unsigned long long &examined)
{
    unsigned c = __ballot_sync(FULL_MASK, lb <= (unsigned)(best >> 32));
    while (c) {
        const int l = __ffs(c) - 1;
        c &= c - 1u;
        if (__shfl_sync(FULL_MASK, lb, l) > (unsigned)(best >> 32))
            continue;   // the bound was overtaken by a closer point
        const unsigned a = __shfl_sync(FULL_MASK, ra, l), b = __shfl_sync(FULL_MASK, rb, l);
        best = scan_run(bpts, a, b, s, lane, best, examined);
    }
    return best;
}

// Lane `sub` of a group of G lanes: its part of the run [a, b) (GROUP_AHEAD
// loads in flight); the group's minimum is the run's.
constexpr int GROUP_AHEAD = 8;

__device__ __forceinline__ unsigned long long group_scan(const float4 *__restrict__ pts, unsigned a, unsigned b,
                                                         float3 s, int sub, int G)
{
    unsigned long long best = ~0ull;
    for (unsigned i = a + (unsigned)sub; i < b; i += (unsigned)(GROUP_AHEAD * G)) {
        float4 q[GROUP_AHEAD];
#pragma unroll
        for (int u = 0; u < GROUP_AHEAD; ++u)   // (past the end: the run's last point again)
            q[u] = __ldg(pts + min(i + (unsigned)(u * G), b - 1u));
#pragma unroll
        for (int u = 0; u < GROUP_AHEAD; ++u)
            best = umin64(best, nn_key(dist2(s, q[u]), __float_as_int(q[u].w)));
    }
    return best;
}

constexpr int SB_CACHED = 4;   // super-brick records kept in registers: 32 per chunk

// The global search of one query s by the whole warp (every lane calls it
// with the same s; every lane gets the result key).  One grid's levels:
// brick records bbox (their w fields: point ranges in bpts), `ns`
// super-brick records sb_box (w fields: brick-record ranges), and the `no`
// target points outside the grid (indices into tgt); tgt holds all n_tgt
// target points.  `examined` counts the candidates (the same on every lane).
// `best` (the same on every lane): a known point's key, or ~0.
__device__ __forceinline__ unsigned long long global_search(float3 s, const float4 *__restrict__ bpts,
                                                            const float4 *__restrict__ bbox,
                                                            const float4 *__restrict__ sb_box, int ns,
                                                            const float4 *__restrict__ tgt, int n_tgt,
                                                            const int *__restrict__ outside, int no, int lane,
                                                            unsigned long long &examined,
                                                            unsigned long long best = ~0ull)
{
    if (!(isfinite(s.x) && isfinite(s.y) && isfinite(s.z))) {
        for (int j = lane; j < n_tgt; j += 32)
            best = umin64(best, nn_key(dist2(s, __ldg(tgt + j)), j));
        examined += (unsigned long long)n_tgt;
        return warp_min_key(best);
    }
    if (ns > 0) {
        // (1) super-brick bounds (the first SB_CACHED chunks kept in
        //     registers; ranges are fetched from L1 when a record is
        //     picked), the nearest super-brick S0 ...
        unsigned sl[SB_CACHED];
        unsigned lmin = 0xffffffffu;
        int kmin = lane;
#pragma unroll
        for (int t = 0; t < SB_CACHED; ++t) {
            const int k = 32 * t + lane;
            sl[t] = 0xffffffffu;
            if (k < ns)
                sl[t] = box_bound(sb_box, k, s);
            if (sl[t] < lmin) {
                lmin = sl[t];
                kmin = k;
            }
        }
        for (int k = 32 * SB_CACHED + lane; k < ns; k += 32) {
            const unsigned lb = box_bound(sb_box, k, s);
            if (lb < lmin) {
                lmin = lb;
                kmin = k;
            }
        }
        const int s0 = min(warp_argmin(lmin, kmin), ns - 1);
        uint2 r0 = box_range(sb_box, s0);
        // ... its bricks' bounds (at most 64: two chunks, kept), and the
        //     nearest brick K0 in it, scanned first for a first distance
        unsigned bl[2];
        unsigned bmin = 0xffffffffu;
        int bk = lane;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int k = 32 * t + lane;   // relative to the super-brick's first brick
            bl[t] = (int)r0.x + k < (int)r0.y ? box_bound(bbox, (int)r0.x + k, s) : 0xffffffffu;
            if (bl[t] < bmin) {
                bmin = bl[t];
                bk = k;
            }
        }
        int k0 = min(warp_argmin(bmin, bk), (int)(r0.y - r0.x) - 1);
        {
            const uint2 pr = box_range(bbox, (int)r0.x + k0);
            if (box_bound(bbox, (int)r0.x + k0, s) <= (unsigned)(best >> 32))   // (a seed may rule it out)
                best = scan_run(bpts, pr.x, pr.y, s, lane, best, examined);
        }
        // (2) best first: the unvisited super-brick of smallest bound
        //     while that bound is <= D, and in it the unvisited brick
        //     of smallest bound while that bound is <= D
#pragma unroll
        for (int t = 0; t < SB_CACHED; ++t)
            if (32 * t + lane == s0)
                sl[t] = 0xffffffffu;
        if ((k0 & 31) == lane) {   // K0 is done
            if (k0 < 32)
                bl[0] = 0xffffffffu;
            else
                bl[1] = 0xffffffffu;
        }
        for (;;) {
            // bricks of the current super-brick (first r0.x), nearest first
            for (;;) {
                const bool first = bl[0] <= bl[1];
                const unsigned v = first ? bl[0] : bl[1];
                const unsigned mn = __reduce_min_sync(FULL_MASK, v);
                if (mn > (unsigned)(best >> 32))
                    break;
                const int w = __ffs(__ballot_sync(FULL_MASK, v == mn)) - 1;
                const int rel = __shfl_sync(FULL_MASK, first ? lane : 32 + lane, w);
                if (lane == w) {
                    if (first)
                        bl[0] = 0xffffffffu;
                    else
                        bl[1] = 0xffffffffu;
                }
                const uint2 pr = box_range(bbox, (int)r0.x + rel);
                best = scan_run(bpts, pr.x, pr.y, s, lane, best, examined);
            }
            // the next super-brick
            unsigned v = 0xffffffffu;
            int vk = lane;
#pragma unroll
            for (int t = 0; t < SB_CACHED; ++t)
                if (sl[t] < v) {
                    v = sl[t];
                    vk = 32 * t + lane;
                }
            const unsigned mn = __reduce_min_sync(FULL_MASK, v);
            if (mn > (unsigned)(best >> 32))
                break;
            const int w = __ffs(__ballot_sync(FULL_MASK, v == mn)) - 1;
            const int sk = __shfl_sync(FULL_MASK, vk, w);
#pragma unroll
            for (int t = 0; t < SB_CACHED; ++t)
                if (lane == w && 32 * t + lane == sk)
                    sl[t] = 0xffffffffu;
            r0 = box_range(sb_box, sk);
#pragma unroll
            for (int t = 0; t < 2; ++t) {   // at most 64 bricks in a super-brick
                const int k = (int)r0.x + 32 * t + lane;
                bl[t] = k < (int)r0.y ? box_bound(bbox, k, s) : 0xffffffffu;
            }
        }
        // super-bricks past the cached chunks, in index order
        for (int c0 = 32 * SB_CACHED; c0 < ns; c0 += 32) {
            unsigned lbs = 0xffffffffu, ra = 0u, rb = 0u;
            if (c0 + lane < ns)
                load_rec(sb_box, c0 + lane, s, lbs, ra, rb);
            unsigned cs = __ballot_sync(FULL_MASK, lbs <= (unsigned)(best >> 32));
            while (cs) {
                const int l = __ffs(cs) - 1;
                cs &= cs - 1u;
                if (__shfl_sync(FULL_MASK, lbs, l) > (unsigned)(best >> 32))
                    continue;   // the bound was overtaken by a closer point
                const unsigned xa = __shfl_sync(FULL_MASK, ra, l), xb = __shfl_sync(FULL_MASK, rb, l);
                for (int kb = (int)xa; kb < (int)xb; kb += 32) {
                    const int k = kb + lane;
                    unsigned lbb = 0xffffffffu, pa = 0u, pb = 0u;
                    if (k < (int)xb)
                        load_rec(bbox, k, s, lbb, pa, pb);
                    best = scan_chunk(bpts, lbb, pa, pb, s, lane, best, examined);
                }
            }
        }
    }
    // (3) target points outside the grid
    for (int k = lane; k < no; k += 32) {
        const int j = __ldg(outside + k);
        best = umin64(best, nn_key(dist2(s, __ldg(tgt + j)), j));
    }
    examined += (unsigned long long)no;
    return warp_min_key(best);
}

}  // namespace vicp
