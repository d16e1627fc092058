// vicp_batch.cu -- batched registration of many pairs over one pooled store
// (layouts in vicp_batch.h).  The grid build of every pair (Alg. 1, Alg. 2,
// the brick levels of the global search, Alg. 3) runs as a handful of
// launches over all pairs at once, and each ICP iteration of every pair
// (Alg. 4 and the update of Eq. 1) is one persistent launch.
//
// The iteration kernel is cooperative: all its blocks are resident together
// and pass one to three grid-wide barriers.
//   phase 1  each warp takes (pair, tile) items as they come: the localised search
//            of the tile's points (a lane per point), the near global queries
//            among them (vicp_search.cuh) from a list in the warp's shared
//            memory, and the tile's sums of what is answered by then; far
//            queries and dense segments are listed for phase 2 (one global
//            atomic per tile and list);
//   phase 2  all warps share out the listed queries of all pairs (dense
//            segments by groups of lanes, a far query by a warp);
//   phase 3  what phase 2 answered joins the sums of its tiles (listed, a warp
//            each); then a block per pair adds the pair's tiles in a fixed
//            order and solves Eq. 1 for that pair, so every pair's update is
//            bit-identical from run to run.
// Phase 2 and the first half of phase 3, with a barrier each, are left out
// when nothing was listed.
// A tile is a warp's own: no block barrier, and no list or match that goes
// through global memory for the points that phase 1 answers.  (With items of
// a block, its barriers between dependent loads left an item of 512 points
// 10 us in phase 1 and 13 us in a phase 3 that read every match again:
// 140 and 190 us of the 560 us an iteration of 256 pairs took.)
// The barriers wait with a time limit (one second): a block that gives up
// sets DEVERR_TIMEOUT and leaves the kernel.
#include <algorithm>

#include "vicp_batch.h"
#include "vicp_df.cuh"
#include "vicp_f64.cuh"
#include "vicp_dilate.cuh"
#include "vicp_launch.h"
#include "vicp_search.cuh"

namespace vicp {

// ---------------------------------------------------------------------------
// Per-pair bounding boxes: one block per 256-point tile; warp-reduced bounds
// merged with one atomic per axis, bound and warp.  bbox: [3P] minima then
// [3P] maxima (order-preserving images).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(BATCH_TILE) k_batch_bbox(const float4 *__restrict__ pts,
                                                           const BatchItem *__restrict__ items, int P,
                                                           unsigned *__restrict__ bbox)
{
    pdl_begin();
    const BatchItem it = items[blockIdx.x];
    const int j = it.i0 + threadIdx.x;
    const float inf = __int_as_float(0x7f800000);
    float lo[3] = {inf, inf, inf}, hi[3] = {-inf, -inf, -inf};
    if (j < it.i1) {
        const float4 q = __ldg(pts + j);
        lo[0] = fminf(lo[0], q.x); hi[0] = fmaxf(hi[0], q.x);
        lo[1] = fminf(lo[1], q.y); hi[1] = fmaxf(hi[1], q.y);
        lo[2] = fminf(lo[2], q.z); hi[2] = fmaxf(hi[2], q.z);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[a] = fminf(lo[a], __shfl_xor_sync(FULL_MASK, lo[a], o));
            hi[a] = fmaxf(hi[a], __shfl_xor_sync(FULL_MASK, hi[a], o));
        }
    }
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            atomicMin(bbox + 3 * it.pair + a, float_to_ordered(lo[a]));
            atomicMax(bbox + 3 * P + 3 * it.pair + a, float_to_ordered(hi[a]));
        }
    }
}

cudaError_t launch_batch_bbox(const float4 *pts, const BatchItem *items, int n_items, int P, unsigned *bbox,
                              cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(bbox, 0xff, 3 * (size_t)P * sizeof(unsigned), st);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(bbox + 3 * P, 0x00, 3 * (size_t)P * sizeof(unsigned), st);
    if (e != cudaSuccess)
        return e;
    return launch_kernel(k_batch_bbox, dim3(n_items), dim3(BATCH_TILE), 0, st, pts, items, P, bbox);
}

// ---------------------------------------------------------------------------
// VOH over all pairs: as the single-grid histogram, with a block per tile of
// one pair.  Keys are the pair's own; counts, occupancy bits and the scan's
// tile totals are indexed by the pooled voxel vbase + key, brick counts by
// bbase + brick.  All lanes of a warp belong to one pair, so grouping by the
// local key groups by the pooled one.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(BATCH_TILE) k_batch_histogram(const float4 *__restrict__ pts,
                                                                const BatchItem *__restrict__ items,
                                                                const BatchPair *__restrict__ pairs,
                                                                int *__restrict__ keys, unsigned *__restrict__ counts,
                                                                unsigned *__restrict__ bcounts,
                                                                unsigned *__restrict__ occ,
                                                                unsigned *__restrict__ tile_sum,
                                                                DevCtl *__restrict__ ctl)
{
    pdl_begin();
    if (blockIdx.x == 0 && threadIdx.x == 0)
        ctl->scan_epoch = ctl->scan_epoch + 1u;
    const BatchItem it = items[blockIdx.x];
    const GridGeom g = pairs[it.pair].g;
    const int vbase = (int)pairs[it.pair].vbase;
    const int bbase = pairs[it.pair].bbase;
    const int j = it.i0 + threadIdx.x;
    int key = -2, bk = -2;   // lanes past the end match only each other and add nothing
    if (j < it.i1) {
        const float4 q = __ldg(pts + j);
        int ix, iy, iz;
        if (voxel_coords(g, q.x, q.y, q.z, ix, iy, iz)) {
            key = ix + g.nx * (iy + g.ny * iz);
            bk = brick_key(g, ix, iy, iz);
        } else {
            key = bk = -1;
        }
        keys[j] = key;
    }
    const int lane = threadIdx.x & 31;
    const int gv = key >= 0 ? vbase + key : -1;
    const unsigned peers = __match_any_sync(FULL_MASK, key);
    if (key >= 0 && lane == __ffs(peers) - 1)
        atomicAdd(counts + gv, (unsigned)__popc(peers));
    const unsigned bpeers = __match_any_sync(FULL_MASK, bk);
    if (bk >= 0 && lane == __ffs(bpeers) - 1)
        atomicAdd(bcounts + bbase + bk, (unsigned)__popc(bpeers));
    const int word = key >= 0 ? (gv >> 5) : -2;
    const unsigned wpeers = __match_any_sync(FULL_MASK, word);
    const unsigned wbits = __reduce_or_sync(wpeers, key >= 0 ? 1u << (gv & 31) : 0u);
    if (word >= 0 && lane == __ffs(wpeers) - 1)
        atomicOr(occ + word, wbits);
    const int tile = key >= 0 ? (gv / SCAN_TILE) : -2;
    const unsigned tpeers = __match_any_sync(FULL_MASK, tile);
    if (tile >= 0 && lane == __ffs(tpeers) - 1)
        atomicAdd(tile_sum + tile, (unsigned)__popc(tpeers));
}

cudaError_t launch_batch_histogram(const float4 *pts, const BatchItem *items, int n_items, const BatchPair *pairs,
                                   int *keys, unsigned *counts, unsigned *bcounts, unsigned *occ, unsigned *tile_sum,
                                   DevCtl *ctl, cudaStream_t st)
{
    return launch_kernel(k_batch_histogram, dim3(n_items), dim3(BATCH_TILE), 0, st, pts, items, pairs, keys, counts,
                         bcounts, occ, tile_sum, ctl);
}

// ---------------------------------------------------------------------------
// Brick offsets, one block per pair: the pair's brick counts scanned
// together with their non-empty flags (as the single-grid brick scan), from
// the pair's first position in the pooled store (off[vbase]).  Brick slots
// are the pair's own, stored at bbase + slot; list holds the pair's own
// brick index, bslot the pooled slot.
// ---------------------------------------------------------------------------
constexpr int BBS_THREADS = 1024;
constexpr int BBS_PER = 8;   // bricks per thread and round

__global__ void __launch_bounds__(BBS_THREADS) k_batch_brick_scan(const unsigned *__restrict__ bcounts,
                                                                  const BatchPair *__restrict__ pairs,
                                                                  const unsigned *__restrict__ off,
                                                                  unsigned *__restrict__ boff, int *__restrict__ list,
                                                                  uint2 *__restrict__ range, int *__restrict__ bslot,
                                                                  uint4 *__restrict__ boxord,
                                                                  BatchState *__restrict__ state)
{
    pdl_begin();
    __shared__ unsigned long long s_w[BBS_THREADS / 32];
    __shared__ unsigned long long s_carry;
    const int p = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const GridGeom g = pairs[p].g;
    const int bbase = pairs[p].bbase;
    const int nbt = brick_slots(g);
    if (tid == 0)
        s_carry = (unsigned long long)__ldg(off + pairs[p].vbase);   // slot count 0, first position
    __syncthreads();
    for (int c0 = 0; c0 < nbt; c0 += BBS_THREADS * BBS_PER) {
        // thread t owns the contiguous bricks [c0 + t*PER, c0 + t*PER + PER)
        unsigned c[BBS_PER];
        unsigned long long sum = 0ull;
#pragma unroll
        for (int k = 0; k < BBS_PER; ++k) {
            const int b = c0 + tid * BBS_PER + k;
            c[k] = b < nbt ? __ldg(bcounts + bbase + b) : 0u;
        }
#pragma unroll
        for (int k = 0; k < BBS_PER; ++k)
            sum += (unsigned long long)c[k] | ((unsigned long long)(c[k] != 0u) << 32);
        unsigned long long incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long y = __shfl_up_sync(FULL_MASK, incl, d);
            if (lane >= d)
                incl += y;
        }
        if (lane == 31)
            s_w[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const unsigned long long w = s_w[lane];
            unsigned long long wi = w;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const unsigned long long y = __shfl_up_sync(FULL_MASK, wi, d);
                if (lane >= d)
                    wi += y;
            }
            s_w[lane] = wi - w;
        }
        __syncthreads();
        unsigned long long run = s_carry + s_w[warp] + (incl - sum);
#pragma unroll
        for (int k = 0; k < BBS_PER; ++k) {
            const int b = c0 + tid * BBS_PER + k;
            if (b < nbt) {
                const unsigned start = (unsigned)run;
                boff[bbase + b] = start;
                if (c[k]) {
                    const int slot = bbase + (int)(run >> 32);
                    list[slot] = b;
                    range[slot] = make_uint2(start, start + c[k]);
                    bslot[bbase + b] = slot;
                    boxord[2 * slot] = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0u);   // min
                    boxord[2 * slot + 1] = make_uint4(0u, 0u, 0u, 0u);                          // max
                }
                run += (unsigned long long)c[k] | ((unsigned long long)(c[k] != 0u) << 32);
            }
        }
        __syncthreads();
        if (tid == BBS_THREADS - 1)
            s_carry = run;
        __syncthreads();
    }
    if (tid == 0)
        state[p].n_bricks = (int)(s_carry >> 32);
}

cudaError_t launch_batch_brick_scan(const unsigned *bcounts, const BatchPair *pairs, int P, const unsigned *off,
                                    unsigned *boff, int *list, uint2 *range, int *bslot, uint4 *boxord,
                                    BatchState *state, cudaStream_t st)
{
    return launch_kernel(k_batch_brick_scan, dim3(P), dim3(BBS_THREADS), 0, st, bcounts, pairs, off, boff, list, range,
                         bslot, boxord, state);
}

// ---------------------------------------------------------------------------
// VDMA over all pairs: as the single-grid scatter, a block per tile of one
// pair.  Segment slots come from the pooled voxel vbase + key; the stored
// index (ids, and the w field of csr and bpts) is the pair's own; target
// points outside the pair's grid are listed at outside + tbase.  Zeroes the
// scan's tile totals for the next build.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(BATCH_TILE) k_batch_scatter(const float4 *__restrict__ pts,
                                                              const int *__restrict__ keys,
                                                              const BatchItem *__restrict__ items,
                                                              const BatchPair *__restrict__ pairs, int n_total,
                                                              const unsigned *__restrict__ off,
                                                              unsigned *__restrict__ counts,
                                                              const unsigned *__restrict__ boff,
                                                              unsigned *__restrict__ bcounts,
                                                              const int *__restrict__ bslot,
                                                              unsigned *__restrict__ boxord, int *__restrict__ ids,
                                                              float4 *__restrict__ csr, float4 *__restrict__ bpts,
                                                              int *__restrict__ outside,
                                                              unsigned *__restrict__ tile_sum, int n_tiles,
                                                              BatchState *__restrict__ state,
                                                              DevCtl *__restrict__ ctl)
{
    pdl_begin();
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_tiles; t += gridDim.x * blockDim.x)
        tile_sum[t] = 0u;
    const BatchItem it = items[blockIdx.x];
    const GridGeom g = pairs[it.pair].g;
    const int vbase = (int)pairs[it.pair].vbase;
    const int bbase = pairs[it.pair].bbase;
    const int tbase = pairs[it.pair].tbase;
    const int j = it.i0 + threadIdx.x;
    const int jl = it.l0 + threadIdx.x;   // the pair's own index
    const int lane = threadIdx.x & 31;
    const int key = (j < it.i1) ? __ldg(keys + j) : -2;
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    int bk = key;
    if (key >= 0) {
        q = __ldg(pts + j);
        int ix, iy, iz;
        bk = voxel_coords(g, q.x, q.y, q.z, ix, iy, iz) ? brick_key(g, ix, iy, iz) : -1;
        q.w = __int_as_float(jl);
    }
    {
        const unsigned peers = __match_any_sync(FULL_MASK, key);
        const int leader = __ffs(peers) - 1;
        const unsigned rank = __popc(peers & lanemask_lt());
        const unsigned cnt = __popc(peers);
        unsigned old = 0u;
        if (lane == leader) {
            if (key >= 0)
                old = atomicSub(counts + vbase + key, cnt);
            else if (key == -1)
                old = (unsigned)atomicAdd(&state[it.pair].n_outside, (int)cnt);
        }
        old = __shfl_sync(FULL_MASK, old, leader);
        if (key >= 0) {
            const unsigned pos = __ldg(off + vbase + key) + old - 1u - rank;
            if (pos < (unsigned)n_total) {
                ids[pos] = jl;
                csr[pos] = q;
            } else {
                atomicOr(&ctl->err, DEVERR_BOUNDS);
            }
        } else if (key == -1) {
            outside[tbase + old + rank] = jl;
        }
    }
    {
        const unsigned peers = __match_any_sync(FULL_MASK, bk);
        const int leader = __ffs(peers) - 1;
        const unsigned rank = __popc(peers & lanemask_lt());
        const unsigned ox = float_to_ordered(q.x), oy = float_to_ordered(q.y), oz = float_to_ordered(q.z);
        const unsigned mnx = __reduce_min_sync(peers, ox), mny = __reduce_min_sync(peers, oy),
                       mnz = __reduce_min_sync(peers, oz);
        const unsigned mxx = __reduce_max_sync(peers, ox), mxy = __reduce_max_sync(peers, oy),
                       mxz = __reduce_max_sync(peers, oz);
        unsigned old = 0u;
        if (lane == leader && bk >= 0) {
            old = atomicSub(bcounts + bbase + bk, (unsigned)__popc(peers));
            unsigned *b = boxord + 8 * __ldg(bslot + bbase + bk);
            atomicMin(b + 0, mnx);
            atomicMin(b + 1, mny);
            atomicMin(b + 2, mnz);
            atomicMax(b + 4, mxx);
            atomicMax(b + 5, mxy);
            atomicMax(b + 6, mxz);
        }
        old = __shfl_sync(FULL_MASK, old, leader);
        if (bk >= 0) {
            const unsigned pos = __ldg(boff + bbase + bk) + old - 1u - rank;
            if (pos < (unsigned)n_total)
                bpts[pos] = q;
            else
                atomicOr(&ctl->err, DEVERR_BOUNDS);
        }
    }
}

cudaError_t launch_batch_scatter(const float4 *pts, const int *keys, const BatchItem *items, int n_items,
                                 const BatchPair *pairs, int n_total, const unsigned *off, unsigned *counts,
                                 const unsigned *boff, unsigned *bcounts, const int *bslot, unsigned *boxord, int *ids,
                                 float4 *csr, float4 *bpts, int *outside, unsigned *tile_sum, int n_tiles,
                                 BatchState *state, DevCtl *ctl, cudaStream_t st)
{
    return launch_kernel(k_batch_scatter, dim3(n_items), dim3(BATCH_TILE), 0, st, pts, keys, items, pairs, n_total,
                         off, counts, boff, bcounts, bslot, boxord, ids, csr, bpts, outside, tile_sum, n_tiles, state,
                         ctl);
}

// ---------------------------------------------------------------------------
// Brick and super-brick records of every pair, one block per pair (as the
// single-grid kernel, on the pair's slots bbase..; super-brick records at
// sbbase.. carry the pair's own brick-record ranges).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_batch_brick_boxes(const uint4 *__restrict__ boxord,
                                                           const int *__restrict__ list,
                                                           const uint2 *__restrict__ range,
                                                           const BatchPair *__restrict__ pairs,
                                                           BatchState *__restrict__ state, float4 *__restrict__ box,
                                                           float4 *__restrict__ sb_box)
{
    pdl_begin();
    const int p = blockIdx.x;
    const int bbase = pairs[p].bbase, sbbase = pairs[p].sbbase;
    const int nb = state[p].n_bricks;
    const uint4 *bo = boxord + 2 * bbase;
    const int *li = list + bbase;
    const uint2 *ra = range + bbase;
    float4 *bx = box + 2 * bbase;
    for (int k = threadIdx.x; k < nb; k += blockDim.x) {
        const uint4 lo = bo[2 * k], hi = bo[2 * k + 1];
        const uint2 r = ra[k];
        bx[2 * k] = make_float4(ordered_to_float(lo.x), ordered_to_float(lo.y), ordered_to_float(lo.z),
                                __uint_as_float(r.x));
        bx[2 * k + 1] = make_float4(ordered_to_float(hi.x), ordered_to_float(hi.y), ordered_to_float(hi.z),
                                    __uint_as_float(r.y));
        const int sb = __ldg(li + k) / SUPER_BRICKS;
        if (k == 0 || __ldg(li + k - 1) / SUPER_BRICKS != sb) {
            uint4 l = lo, h = hi;
            int e = k + 1;
            while (e < nb && __ldg(li + e) / SUPER_BRICKS == sb) {
                const uint4 bl = bo[2 * e], bh = bo[2 * e + 1];
                l = make_uint4(min(l.x, bl.x), min(l.y, bl.y), min(l.z, bl.z), 0u);
                h = make_uint4(max(h.x, bh.x), max(h.y, bh.y), max(h.z, bh.z), 0u);
                ++e;
            }
            const int slot = sbbase + atomicAdd(&state[p].n_super, 1);
            sb_box[2 * slot] = make_float4(ordered_to_float(l.x), ordered_to_float(l.y), ordered_to_float(l.z),
                                           __uint_as_float((unsigned)k));
            sb_box[2 * slot + 1] = make_float4(ordered_to_float(h.x), ordered_to_float(h.y), ordered_to_float(h.z),
                                               __uint_as_float((unsigned)e));
        }
    }
}

cudaError_t launch_batch_brick_boxes(const uint4 *boxord, const int *list, const uint2 *range,
                                     const BatchPair *pairs, int P, BatchState *state, float4 *box, float4 *sb_box,
                                     cudaStream_t st)
{
    return launch_kernel(k_batch_brick_boxes, dim3(P), dim3(256), 0, st, boxord, list, range, pairs, state, box,
                         sb_box);
}

// ---------------------------------------------------------------------------
// Dilation of every pair's grid: the single-grid passes (vicp_dilate.cuh)
// over the concatenated units of all pairs.  A warp finds the pair of its
// unit by binary search in the pairs' first-unit table (kept in shared
// memory for up to BATCH_SMEM_PAIRS pairs) and runs the unit on the pair's
// slices of the pooled arrays.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int find_pair(const int *starts, int P, int u)
{
    int lo = 0, hi = P - 1;   // starts[lo] <= u < starts[hi + 1]
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (starts[mid] <= u)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ const int *stage_starts(const int *starts, int P, int *s_buf)
{
    if (P + 1 > BATCH_SMEM_PAIRS)
        return starts;
    for (int k = threadIdx.x; k <= P; k += blockDim.x)
        s_buf[k] = __ldg(starts + k);
    __syncthreads();
    return s_buf;
}

template <class W>
__global__ void __launch_bounds__(dil::THREADS) k_batch_dilate_xy(const unsigned *__restrict__ occ,
                                                                  const BatchPair *__restrict__ pairs, int P,
                                                                  const int *__restrict__ ustart, int L,
                                                                  typename W::Stored *__restrict__ inter,
                                                                  unsigned *__restrict__ rows)
{
    pdl_begin();
    extern __shared__ int s_starts[];
    const int *starts = stage_starts(ustart, P, s_starts);
    const int units = __ldg(ustart + P);
    for (int u = blockIdx.x * dil::WARPS + (threadIdx.x >> 5); u < units; u += gridDim.x * dil::WARPS) {
        const int p = find_pair(starts, P, u);
        const GridGeom g = pairs[p].g;
        const long long vb = pairs[p].vbase;
        const int nxb = (g.nx + dil::UX - 1) / dil::UX, nyb = (g.ny + dil::UY - 1) / dil::UY;
        const int u0 = starts[p];
        dil::dilate_xy_unit<W>(u - u0, occ + (vb >> 5), (g.V + 31) / 32, g, L, nxb, nyb, inter + vb, rows + u0);
    }
}

template <class W>
__global__ void __launch_bounds__(dil::THREADS) k_batch_dilate_z(const typename W::Stored *__restrict__ inter,
                                                                 const unsigned *__restrict__ rows,
                                                                 unsigned char *__restrict__ dirty,
                                                                 const BatchPair *__restrict__ pairs, int P,
                                                                 const int *__restrict__ ustart_xy,
                                                                 const int *__restrict__ ustart, int L,
                                                                 int *__restrict__ root,
                                                                 unsigned char *__restrict__ ring)
{
    pdl_begin();
    extern __shared__ int s_starts[];
    const int *starts = stage_starts(ustart, P, s_starts);
    const int units = __ldg(ustart + P);
    for (int u = blockIdx.x * dil::WARPS + (threadIdx.x >> 5); u < units; u += gridDim.x * dil::WARPS) {
        const int p = find_pair(starts, P, u);
        const GridGeom g = pairs[p].g;
        const long long vb = pairs[p].vbase;
        const int nxb = (g.nx + dil::UX - 1) / dil::UX, nyb = (g.ny + dil::UY - 1) / dil::UY;
        const int u0 = starts[p];
        dil::dilate_z_unit<W>(u - u0, inter + vb, rows + __ldg(ustart_xy + p),
                              dil::DenseLabels{dirty + u0, root + vb, ring + vb}, g, L, nxb, nyb);
    }
}

template <typename K>
static int resident_blocks_of(K kernel, int threads, size_t smem)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    return sms * per_sm;
}

template <class W>
static cudaError_t run_batch_dilate(const unsigned *occ, const BatchPair *pairs, int P, const int *ustart_xy,
                                    const int *ustart_z, int L, void *inter, unsigned *rows, unsigned char *dirty,
                                    int *root, unsigned char *ring, int units_xy, int units_z, cudaStream_t st)
{
    using S = typename W::Stored;
    const size_t smem = P + 1 <= BATCH_SMEM_PAIRS ? (size_t)(P + 1) * sizeof(int) : 0;
    const int xy_blocks = resident_blocks_of(k_batch_dilate_xy<W>, dil::THREADS, smem);
    const int z_blocks = resident_blocks_of(k_batch_dilate_z<W>, dil::THREADS, smem);
    cudaError_t e = launch_kernel(k_batch_dilate_xy<W>, dim3(min(xy_blocks, (units_xy + dil::WARPS - 1) / dil::WARPS)),
                                  dim3(dil::THREADS), smem, st, occ, pairs, P, ustart_xy, L, static_cast<S *>(inter),
                                  rows);
    if (e != cudaSuccess)
        return e;
    return launch_kernel(k_batch_dilate_z<W>, dim3(min(z_blocks, (units_z + dil::WARPS - 1) / dil::WARPS)),
                         dim3(dil::THREADS), smem, st, static_cast<const S *>(inter), rows, dirty, pairs, P, ustart_xy,
                         ustart_z, L, root, ring);
}

cudaError_t launch_batch_dilate(const unsigned *occ, const BatchPair *pairs, int P, const int *ustart_xy,
                                const int *ustart_z, int L, void *inter, unsigned *rows, unsigned char *dirty,
                                int *root, unsigned char *ring, cudaStream_t st)
{
    // unit totals: read back by the caller would cost a synchronisation, so
    // the grids are sized from the resident block count alone
    const int big = 1 << 30;
    if (L <= dil::L_COMPACT_MAX)
        return run_batch_dilate<dil::Words16>(occ, pairs, P, ustart_xy, ustart_z, L, inter, rows, dirty, root, ring,
                                              big, big, st);
    return run_batch_dilate<dil::Words32>(occ, pairs, P, ustart_xy, ustart_z, L, inter, rows, dirty, root, ring, big,
                                          big, st);
}

// ---------------------------------------------------------------------------
// Grid-wide barrier of the cooperative iteration kernel, with a time limit.
// One thread per block arrives (atomic ticket after a fence that publishes
// the block's writes); the last one resets the ticket and advances the
// generation with a release store; the others poll the generation with
// acquire loads.  Returns false, with DEVERR_TIMEOUT set, when the
// generation has not moved for BARRIER_LIMIT_NS.
// ---------------------------------------------------------------------------
constexpr unsigned long long BARRIER_LIMIT_NS = 1000000000ull;

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_u32(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ bool grid_barrier(DevCtl *ctl, int *s_flag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned gen = ld_acquire_u32(&ctl->bar_gen);
        __threadfence();
        const unsigned arrived = atomicAdd(&ctl->bar_count, 1u);
        if (arrived == gridDim.x - 1) {
            ctl->bar_count = 0u;
            st_release_u32(&ctl->bar_gen, gen + 1u);
        } else {
            const unsigned long long t0 = globaltimer_ns();
            unsigned polls = 0;
            while (ld_acquire_u32(&ctl->bar_gen) == gen) {
                __nanosleep(64);
                if ((++polls & 255u) == 0u && globaltimer_ns() - t0 > BARRIER_LIMIT_NS) {
                    atomicOr(&ctl->err, DEVERR_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        *s_flag = ok;
    }
    __syncthreads();
    return *s_flag != 0;
}

// The float pose of a pair, as phase 1 stored it.
__device__ __forceinline__ PoseF load_posef(const float *__restrict__ posef, int pair)
{
    static_assert(sizeof(PoseF) == 48, "PoseF layout");
    const float4 *p = reinterpret_cast<const float4 *>(posef + 12 * pair);
    const float4 a = __ldcg(p), b = __ldcg(p + 1), c = __ldcg(p + 2);
    return PoseF{{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x}, {c.y, c.z, c.w}};
}

// ---------------------------------------------------------------------------
// The sums of phases 1 and 3 in double-float or, for the FP64 variant, in
// doubles (vicp_df.cuh, vicp_f64.cuh): 8 bytes a value either way.
// ---------------------------------------------------------------------------
template <bool F64> struct IterSum;

template <> struct IterSum<false> {
    using T = dfl;
    __device__ static T zero() { return {0.0f, 0.0f}; }
    __device__ static T add(T a, T b) { return df_acc(a, b); }
    __device__ static T shfl_xor(T v, int o) { return df_shfl_xor(v, o); }
    __device__ static T load(const float2 *p)
    {
        const float2 x = __ldcg(p);
        return {x.x, x.y};
    }
    __device__ static void store(float2 *p, T v) { *p = make_float2(v.hi, v.lo); }
    __device__ static void accumulate(T (&acc)[N_SUMS], float3 s, float4 q, const BatchPair *bp)
    {
        accumulate_corr(acc, s, q, make_float3(bp->cx, bp->cy, bp->cz));
    }
    __device__ static bool solve(const T *s_tot, const BatchPair *bp, double *pose, double &rmse)
    {
        return solve_update(s_tot, bp->n_src, make_float3(bp->cx, bp->cy, bp->cz), pose, rmse);
    }
};

template <> struct IterSum<true> {
    using T = double;
    __device__ static T zero() { return 0.0; }
    __device__ static T add(T a, T b) { return a + b; }
    __device__ static T shfl_xor(T v, int o) { return __shfl_xor_sync(FULL_MASK, v, o); }
    __device__ static T load(const float2 *p) { return __ldcg(reinterpret_cast<const double *>(p)); }
    __device__ static void store(float2 *p, T v) { *reinterpret_cast<double *>(p) = v; }
    __device__ static void accumulate(T (&acc)[N_SUMS], float3 s, float4 q, const BatchPair *bp)
    {
        static_assert(N_SUMS == F64_SUMS, "sum layout");
        accumulate_corr_f64(acc, s, q, make_double3((double)bp->cx, (double)bp->cy, (double)bp->cz));
    }
    __device__ static bool solve(const T *s_tot, const BatchPair *bp, double *pose, double &rmse)
    {
        return solve_update_f64(s_tot, bp->n_src, make_double3((double)bp->cx, (double)bp->cy, (double)bp->cz), pose,
                                rmse);
    }
};

// A warp's shared memory: the tile's matches, seeds and lists while it is
// searched, then the lanes' sums laid out for the warp's reduction.
struct WarpTile {
    union {
        struct {
            float pose[12];
            int nn[BATCH_TILE_MAX];      // match of each point; -1: left to phase 2 (or no point)
            float d2[BATCH_TILE_MAX];    // seed of a near query
            unsigned char near[BATCH_TILE_MAX], far[BATCH_TILE_MAX];
        };
        double lanes[N_SUMS][33];        // a row per sum (row stride 33: no bank conflicts either way)
    };
};

// The tile's 16 sums from the lanes' (fixed order): sum k on lanes k and
// k + 16.  The whole warp calls it; w's contents are overwritten.
template <bool F64>
__device__ __forceinline__ typename IterSum<F64>::T tile_sum(const typename IterSum<F64>::T (&acc)[N_SUMS], WarpTile &w)
{
    using S = IterSum<F64>;
    using T = typename S::T;
    static_assert(sizeof(T) == sizeof(double), "sum words");
    const int lane = threadIdx.x & 31;
    T(*rows)[33] = reinterpret_cast<T(*)[33]>(w.lanes);
    __syncwarp();
#pragma unroll
    for (int k = 0; k < N_SUMS; ++k)
        rows[k][lane] = acc[k];
    __syncwarp();
    const int k = lane & 15, h = (lane >> 4) * 16;
    T v = rows[k][h];
#pragma unroll
    for (int t = 1; t < 16; ++t)
        v = S::add(v, rows[k][h + t]);
    v = S::add(v, S::shfl_xor(v, 16));
    __syncwarp();
    return v;
}

// Points of a root segment examined for the seed of a query outside the grid:
// all of them wherever the query can be near (near_seed, whose other factor
// is at least 2), and the first NEAR_SEED of a longer one.  The order of a
// voxel's points in the store varies from build to build.  A seed from some of
// them would decide, by that order, whether the query is near and summed in
// phase 1, or far and summed in phase 3, and the last bits of the pose would
// vary with it (from the first 16: of 24 to 31 of 256 pairs).  256 pairs, 40
// iterations: 25.9 ms from the first 16, 26.0 from all.  (The searches alone
// form no sums.)
constexpr unsigned TILE_SEED = NEAR_WORK / 2;

// The near queries of a tile, 1 to 32 lanes each; returns the candidates
// this lane examined.  (Out of line, it and the sums below spill less and
// are slower: 256 pairs 28.8 ms a batch against 25.9.)
template <bool SEARCH_ONLY>
static __device__ __forceinline__ unsigned near_tile(const BatchIterArgs &a, WarpTile &w, const BatchItem &it, int n_near)
{
    const int lane = threadIdx.x & 31;
    const BatchPair *bp = a.pairs + it.pair;
    const GridGeom g = bp->g;
    const long long vb = bp->vbase;
    const CsrRows rows{a.occ + (vb >> 5), a.off + vb, (unsigned)a.n_stored, a.csr};
    const PoseF P = *reinterpret_cast<const PoseF *>(w.pose);
    const int no = a.state[it.pair].n_outside;
    const int shift = group_shift(n_near, 32, NEAR_SHIFT_MIN), G = 1 << shift, pack = 32 >> shift;
    const int sub = lane & (G - 1);
    unsigned cand = 0u;
    for (int k = 0; k < n_near; k += pack) {
        const int q = k + (lane >> shift);
        const bool on = q < n_near;
        const int l = on ? w.near[q] : 0, i = it.i0 + l;
        float3 s = make_float3(0.0f, 0.0f, 0.0f);
        unsigned long long best = ~0ull;
        if (on) {
            s = transform_pt(P, __ldg(a.src + i));
            best = nn_key(w.d2[l], w.nn[l]);
            for (int o = sub; o < no; o += G) {   // target points outside the grid
                const int j = __ldg(a.outside + bp->tbase + o);
                best = umin64(best, nn_key(dist2(s, __ldg(a.tgt + bp->tbase + j)), j));
            }
            cand += sub == 0 ? (unsigned)no : 0u;
        }
        if (no > 0)
            best = group_min(best, G);
        best = near_search(g, rows, s, best, on, sub, G, cand);
        if (on && sub == 0) {
            w.nn[l] = (int)(unsigned)best;
            if (SEARCH_ONLY) {
                a.nn[i] = (int)(unsigned)best;
                a.d2[i] = __uint_as_float((unsigned)(best >> 32));
            }
        }
    }
    __syncwarp();
    return cand;
}

// The sums of a tile's matches w.nn, stored as item itx's; lane r gets the
// mask of the points 32 r .. 32 r + 31 that have none yet.
template <bool F64>
static __device__ __forceinline__ unsigned sum_tile(const BatchIterArgs &a, WarpTile &w, const BatchItem &it, int itx)
{
    using S = IterSum<F64>;
    using T = typename S::T;
    const int lane = threadIdx.x & 31, n = it.i1 - it.i0;
    const BatchPair *bp = a.pairs + it.pair;
    const PoseF P = *reinterpret_cast<const PoseF *>(w.pose);
    T acc[N_SUMS];
#pragma unroll
    for (int k = 0; k < N_SUMS; ++k)
        acc[k] = S::zero();
    unsigned left = 0u;
#pragma unroll 1
    for (int l0 = 0; l0 < n; l0 += 32) {
        const int l = l0 + lane;
        const int j = l < n ? w.nn[l] : -1;
        if ((unsigned)j < (unsigned)bp->n_tgt)
            S::accumulate(acc, transform_pt(P, __ldg(a.src + it.i0 + l)), __ldg(a.tgt + bp->tbase + j), bp);
        else if (j >= 0)   // no valid match: report, leave it out
            atomicOr(&a.ctl->err, DEVERR_BOUNDS);
        const unsigned m = __ballot_sync(FULL_MASK, l < n && j < 0);
        if (lane == (l0 >> 5))
            left = m;
    }
    const T v = tile_sum<F64>(acc, w);
    if (lane < N_SUMS)
        S::store(a.partials + (size_t)itx * N_SUMS + lane, v);
    return left;
}

// ---------------------------------------------------------------------------
// The iteration kernel (see the top of this file).  Dynamic shared memory: a
// WarpTile per warp.
// ---------------------------------------------------------------------------
template <int TH, int MINB, bool F64, bool SEARCH_ONLY = false, int UNROLL = 1>
__global__ void __launch_bounds__(TH, MINB) k_batch_iter(const __grid_constant__ BatchIterArgs a)
{
    constexpr int WARPS = TH / 32;
    using S = IterSum<F64>;
    using T = typename S::T;
    __shared__ int s_flag;
    __shared__ unsigned long long s_cand, s_queries, s_near, s_glob;   // work counters: one global atomic a block
    extern __shared__ double s_dyn[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    WarpTile &w = reinterpret_cast<WarpTile *>(s_dyn)[warp];
    DevCtl *const ctl = a.ctl;
    // After a barrier gave up, the arrival count no longer matches the
    // blocks in the barrier: the remaining launches of the registration do
    // nothing (the host clears the status and the count).
    if (*(volatile const unsigned *)&ctl->err & DEVERR_TIMEOUT)
        return;
    if (a.test_leave_early && blockIdx.x == 0)
        return;   // the others' first barrier runs out of time (test of the time limit)
    if (tid == 0)
        s_cand = s_queries = s_near = s_glob = 0ull;
    __syncthreads();
    const int n_warps = gridDim.x * WARPS, gw = blockIdx.x * WARPS + warp;

    // ---- phase 1: each warp's tiles: localised and near searches, sums ------
    unsigned cand = 0u, queries = 0u, near_done = 0u, near_cand = 0u;
    // The first tile by position, then whichever is next (the ticket is drawn
    // while the tile before is searched): tiles differ several-fold.
    unsigned ticket = 0u;
    for (int itx = gw; itx < a.n_items;
         itx = a.n_items > n_warps ? n_warps + (int)__shfl_sync(FULL_MASK, ticket, 0) : a.n_items) {
        if (lane == 0 && a.n_items > n_warps)
            ticket = atomicAdd(&ctl->item_next, 1u);
        const BatchItem it = a.items[itx];
        if (!SEARCH_ONLY && __ldcg(&a.state[it.pair].stop))
            continue;
        __syncwarp();   // the last tile's use of w is over
        if (lane < 12) {
            const int r = lane >> 2, c = lane & 3, k = c < 3 ? 3 * r + c : 9 + r;
            const float v = __double2float_rn(__ldcg(a.pose + 16 * it.pair + lane));
            w.pose[k] = v;
            if (it.l0 == 0)   // the pair's first tile: for phase 2
                a.posef[12 * it.pair + k] = v;
        }
        const bool seeds = a.state[it.pair].n_outside <= NEAR_OUTSIDE_MAX;
        const BatchPair *bp = a.pairs + it.pair;
        const GridGeom g = bp->g;
        const long long vb = bp->vbase;
        const CsrRows rows{a.occ + (vb >> 5), a.off + vb, (unsigned)a.n_stored, a.csr};
        __syncwarp();
        const PoseF P = *reinterpret_cast<const PoseF *>(w.pose);
        const int n = it.i1 - it.i0;
        int n_near = 0, n_far = 0;
#pragma unroll UNROLL
        for (int l0 = 0; l0 < n; l0 += 32) {
            const int l = l0 + lane, i = it.i0 + l;
            bool far = false, near = false, heavy = false;
            unsigned x0 = 0u, x1 = 0u;
            if (l < n) {   // (as k_correspond)
                const float3 s = transform_pt(P, __ldg(a.src + i));
                bool inside;
                const int v = nearest_voxel(g, s, inside);
                const int r = v >= 0 ? __ldg(a.root + vb + v) : -1;
                unsigned dense = 0u;
                if (r >= 0) {
                    x0 = __ldg(rows.off + r);
                    x1 = max(x0, min(__ldg(rows.off + r + 1), rows.cap));
                    dense = x1 - x0;
                    if (!inside)   // only a seed
                        x1 = min(x1, x0 + (SEARCH_ONLY || dense > TILE_SEED ? (unsigned)NEAR_SEED : TILE_SEED));
                }
                const bool local = inside && r >= 0;
                cand += local ? dense : 0u;
                heavy = local && dense > HEAVY;
                if (!heavy) {
                    const unsigned long long best = segment_min(rows.csr, x0, x1, s);
                    const float d = __uint_as_float((unsigned)(best >> 32));
                    near = !local && dense && seeds && near_seed(s, d, g.inv_h, dense);
                    far = !local && !near;
                    if (near)
                        w.d2[l] = d;
                    if (far || SEARCH_ONLY) {   // (a far query's seed, or the answer)
                        a.nn[i] = (int)(unsigned)best;
                        a.d2[i] = d;
                    }
                    w.nn[l] = far ? -1 : (int)(unsigned)best;
                } else {
                    w.nn[l] = -1;
                }
            }
            const unsigned nm = __ballot_sync(FULL_MASK, near), fm = __ballot_sync(FULL_MASK, far);
            if (near)
                w.near[n_near + __popc(nm & lanemask_lt())] = (unsigned char)l;
            if (far)
                w.far[n_far + __popc(fm & lanemask_lt())] = (unsigned char)l;
            n_near += __popc(nm);
            n_far += __popc(fm);
            const unsigned hm = __ballot_sync(FULL_MASK, heavy);
            if (hm) {   // dense segments: listed right away
                int slot = lane == 0 ? atomicAdd(&ctl->hv_count, __popc(hm)) : 0;
                slot = __shfl_sync(FULL_MASK, slot, 0) + __popc(hm & lanemask_lt());
                if (heavy) {
                    if (slot < a.list_cap)
                        a.hv_list[slot] = make_int4(it.pair, i, (int)x0, (int)x1);
                    else
                        atomicOr(&ctl->err, DEVERR_BOUNDS);
                }
            }
        }
        queries += (unsigned)n;
        near_done += (unsigned)n_near;
        __syncwarp();
        if (n_far) {   // one global atomic a tile
            int slot0 = lane == 0 ? atomicAdd(&ctl->fb_count, n_far) : 0;
            slot0 = __shfl_sync(FULL_MASK, slot0, 0);
            for (int k = lane; k < n_far; k += 32) {
                if (slot0 + k < a.list_cap)
                    a.fb_list[slot0 + k] = make_int2(it.pair, it.i0 + w.far[k]);
                else
                    atomicOr(&ctl->err, DEVERR_BOUNDS);
            }
        }
        if (n_near)
            near_cand += near_tile<SEARCH_ONLY>(a, w, it, n_near);
        if constexpr (!SEARCH_ONLY) {
            // the sums of the points answered here, and which are left
            const unsigned left = sum_tile<F64>(a, w, it, itx);
            if (__any_sync(FULL_MASK, left != 0u)) {
                if (lane < BATCH_TILE_MAX / 32)
                    a.left[(size_t)itx * (BATCH_TILE_MAX / 32) + lane] = left;
                if (lane == 0)
                    a.open_items[atomicAdd(&ctl->open_count, 1)] = itx;
            }
        }
    }
    {
        const unsigned long long c = warp_sum_u64(cand), gl = warp_sum_u64(near_cand);
        if (lane == 0) {
            if (c)
                atomicAdd(&s_cand, c);
            if (gl)
                atomicAdd(&s_glob, gl);
            if (queries)
                atomicAdd(&s_queries, (unsigned long long)queries);
            if (near_done)
                atomicAdd(&s_near, (unsigned long long)near_done);
        }
    }
    if (!grid_barrier(ctl, &s_flag))
        return;

    // ---- phase 2: dense segments and far queries of all pairs ---------------
    const int F = min(*(volatile int *)&ctl->fb_count, a.list_cap);
    const int Hv = min(*(volatile int *)&ctl->hv_count, a.list_cap);
    if (tid == 0) {
        if (blockIdx.x == 0)
            ctl->item_next = 0u;   // (every tile is taken)
        if (s_cand)
            atomicAdd(&ctl->stat_local_cand, s_cand);
        if (s_queries)
            atomicAdd(&ctl->stat_queries, s_queries);
        if (s_near)
            atomicAdd(&ctl->stat_fallbacks, s_near);
    }
    unsigned long long examined = 0ull;   // far queries: every lane counts the same
    {   // dense segments, 4 to 32 lanes each
        const int shift = group_shift(Hv, n_warps * 32, HEAVY_SHIFT_MIN), G = 1 << shift, pack = 32 >> shift;
        const int sub = lane & (G - 1);
        for (int q0 = (n_warps - 1 - gw) * pack; q0 < Hv; q0 += n_warps * pack) {
            const int q = q0 + (lane >> shift);
            const int4 e = q < Hv ? a.hv_list[q] : make_int4(-1, -1, 0, 0);
            const bool on = (unsigned)e.x < (unsigned)a.n_pairs && (unsigned)e.y < (unsigned)a.list_cap &&
                            e.z <= e.w && (unsigned)e.w <= (unsigned)a.n_stored;
            if (!on && q < Hv)   // a stale entry: skip it, report it
                atomicOr(&ctl->err, DEVERR_BOUNDS);
            unsigned long long best = ~0ull;
            if (on)
                best = group_scan(a.csr, (unsigned)e.z, (unsigned)e.w,
                                  transform_pt(load_posef(a.posef, e.x), __ldg(a.src + e.y)), sub, G);
            best = group_min(best, G);
            if (on && sub == 0) {
                a.nn[e.y] = (int)(unsigned)best;
                a.d2[e.y] = __uint_as_float((unsigned)(best >> 32));
            }
        }
    }
    // far queries: a first chunk per warp, then chunks to whichever warp is
    // free (a ticket per chunk): their costs vary widely, and a fixed share
    // per warp leaves the whole grid waiting at the barrier for the warp
    // that drew the slowest ones
    const int far_chunk = min(max(F / (4 * n_warps), 1), 4);
    for (int q0 = gw * far_chunk; q0 < F;) {
        for (int qi = q0; qi < min(q0 + far_chunk, F); ++qi) {
            const int2 e = a.fb_list[qi];
            if ((unsigned)e.x >= (unsigned)a.n_pairs || (unsigned)e.y >= (unsigned)a.list_cap) {
                if (lane == 0)   // a stale entry: skip it, report it
                    atomicOr(&ctl->err, DEVERR_BOUNDS);
                continue;
            }
            const BatchPair *bp = a.pairs + e.x;
            const float3 s = transform_pt(load_posef(a.posef, e.x), __ldg(a.src + e.y));
            const int tbase = bp->tbase;
            const unsigned long long best = global_search(
                s, a.bpts, a.bbox + 2 * bp->bbase, a.sb_box + 2 * bp->sbbase, a.state[e.x].n_super, a.tgt + tbase,
                bp->n_tgt, a.outside + tbase, a.state[e.x].n_outside, lane, examined,
                nn_key(__ldcg(a.d2 + e.y), __ldcg(a.nn + e.y)));
            __syncwarp();   // every lane has read the seed
            if (lane == 0) {
                a.nn[e.y] = (int)(unsigned)best;
                a.d2[e.y] = __uint_as_float((unsigned)(best >> 32));
            }
        }
        if ((long long)n_warps * far_chunk >= F)
            break;
        if (lane == 0)
            q0 = far_chunk * (n_warps + (int)atomicAdd(&ctl->fb_next, 1u));
        q0 = __shfl_sync(FULL_MASK, q0, 0);
    }
    if (lane == 0 && examined)
        atomicAdd(&s_glob, examined);
    if (F + Hv) {   // (the same in every block: the lists are complete)
        if (!grid_barrier(ctl, &s_flag))
            return;
        if (blockIdx.x == 0 && tid == 0) {   // every block has read the list lengths
            ctl->stat_fallbacks += (unsigned long long)F;
            ctl->fb_count = 0;
            ctl->hv_count = 0;
            ctl->fb_next = 0u;
        }
    } else {
        __syncthreads();
    }
    if (tid == 0 && s_glob)
        atomicAdd(&ctl->stat_global_cand, s_glob);
    if constexpr (SEARCH_ONLY)
        return;

    // ---- phase 3: what phase 2 answered joins its tiles' sums ---------------
    if (F + Hv) {
        const int n_open = min(__ldcg(&ctl->open_count), a.n_items);
        for (int o = gw; o < n_open; o += n_warps) {
            const int itx = __ldcg(a.open_items + o);
            const BatchItem it = a.items[itx];
            const BatchPair *bp = a.pairs + it.pair;
            const unsigned left =
                lane < BATCH_TILE_MAX / 32 ? __ldcg(a.left + (size_t)itx * (BATCH_TILE_MAX / 32) + lane) : 0u;
            const PoseF P = load_posef(a.posef, it.pair);
            T acc[N_SUMS];
#pragma unroll
            for (int k = 0; k < N_SUMS; ++k)
                acc[k] = S::zero();
#pragma unroll 1
            for (int l0 = 0; l0 < it.i1 - it.i0; l0 += 32) {
                const unsigned m = __shfl_sync(FULL_MASK, left, l0 >> 5);
                if (!((m >> lane) & 1u))
                    continue;
                const int i = it.i0 + l0 + lane;
                const int j = __ldcg(a.nn + i);
                if ((unsigned)j < (unsigned)bp->n_tgt)
                    S::accumulate(acc, transform_pt(P, __ldg(a.src + i)), __ldg(a.tgt + bp->tbase + j), bp);
                else   // no valid match: report, leave it out
                    atomicOr(&ctl->err, DEVERR_BOUNDS);
            }
            __syncwarp();
            const T v = tile_sum<F64>(acc, w);
            float2 *part = a.partials + (size_t)itx * N_SUMS;
            if (lane < N_SUMS)
                S::store(part + lane, S::add(S::load(part + lane), v));
        }
        if (!grid_barrier(ctl, &s_flag))
            return;
        if (blockIdx.x == 0 && tid == 0)
            ctl->open_count = 0;
    }

    // ---- and a block per pair adds the pair's tiles in a fixed order and
    // solves: thread t adds sum t % 16 of tiles t / 16, t / 16 + TH / 16, ...;
    // then the groups in order (pairs of them by a shuffle, then the warps) ---
    __shared__ T s_w[WARPS][N_SUMS], s_tot[N_SUMS];
    for (int p = blockIdx.x; p < a.n_pairs; p += gridDim.x) {
        BatchState *stp = a.state + p;
        const int stop = __ldcg(&stp->stop);
        __syncthreads();   // (read by all before it can change; s_w is free)
        if (stop)
            continue;
        const BatchPair *bp = a.pairs + p;
        const int k = tid & 15, n_items = bp->n_items;
        const float2 *p0 = a.partials + (size_t)bp->item0 * N_SUMS + k;
        T v = S::zero();
        for (int b = tid >> 4; b < n_items; b += 8 * (TH / 16)) {   // eight loads in flight
            T x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                x[u] = b + u * (TH / 16) < n_items ? S::load(p0 + (size_t)(b + u * (TH / 16)) * N_SUMS) : S::zero();
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v = S::add(v, x[u]);
        }
        v = S::add(v, S::shfl_xor(v, 16));
        if (lane < N_SUMS)
            s_w[warp][lane] = v;
        __syncthreads();
        if (warp == 0) {
            if (lane < N_SUMS) {
                T t = s_w[0][lane];
#pragma unroll
                for (int q = 1; q < WARPS; ++q)
                    t = S::add(t, s_w[q][lane]);
                s_tot[lane] = t;
            }
            __syncwarp();
            double rmse;
            const bool ok = S::solve(s_tot, bp, a.pose + 16 * p, rmse);
            if (lane == 0) {
                stp->last_rmse = rmse;
                if (!ok) {
                    stp->err |= DEVERR_DEGENERATE;
                    stp->stop = 1;
                    atomicOr(&ctl->err, DEVERR_DEGENERATE);
                } else {
                    const int it = stp->iters;
                    stp->iters = it + 1;
                    if (a.eps > 0.0 && it >= 1 && fabs(rmse - stp->prev_rmse) < a.eps)
                        stp->stop = 1;
                    stp->prev_rmse = rmse;
                }
            }
        }
    }
}

// (Tiles have at most BATCH_TILE_MAX points, fewer where the batch has few: 64
// to 256 differ by under 3% on 256 pairs, and the searches alone prefer 128,
// 64 x 20k points 107 us against 125 with 256.)
const BatchShape BATCH_SHAPES[BATCH_N_SHAPES] = {
    {256, 4, 2},   // 128 registers
    {256, 2, 3},   // 80 registers, more warps per SM (196 bytes of spill stores, 248 of loads)
    {512, 2, 1},   // wide blocks
    {128, 4, 4},   // narrow blocks
    {256, 8, 2},   // as 0
    {256, 2, 4},   // 64 registers (492 bytes of spill stores, 652 of loads)
    {256, 2, 5},   // 48 registers (over 1 KB of either: most of the sums)
};

using IterKernel = void (*)(const BatchIterArgs);

static IterKernel iter_kernel(int shape, BatchMode mode)
{
    const bool f64 = mode == BATCH_FP64;
    if (mode == BATCH_SEARCH)   // without the sums every shape's searches run best with the most warps
        return k_batch_iter<256, 2, false, true, 4>;
    switch (shape) {
    case 0: case 4: return f64 ? k_batch_iter<256, 2, true> : k_batch_iter<256, 2, false>;
    case 1: return f64 ? k_batch_iter<256, 3, true> : k_batch_iter<256, 3, false>;
    case 2: return f64 ? k_batch_iter<512, 1, true> : k_batch_iter<512, 1, false>;
    case 3: return f64 ? k_batch_iter<128, 4, true> : k_batch_iter<128, 4, false>;
    case 5: return f64 ? k_batch_iter<256, 4, true> : k_batch_iter<256, 4, false>;
    case 6: return f64 ? k_batch_iter<256, 5, true> : k_batch_iter<256, 5, false>;
    }
    return nullptr;
}

static int iter_threads(int shape, BatchMode mode) { return mode == BATCH_SEARCH ? 256 : BATCH_SHAPES[shape].threads; }
static size_t iter_smem(int threads) { return (size_t)(threads / 32) * sizeof(WarpTile); }

int batch_tile_points(int shape, int blocks, long long m)
{
    // whole rounds of all warps: k tiles a warp, of as few points as k needs
    const long long lanes = std::max((long long)blocks * BATCH_SHAPES[shape].threads, 32ll);
    const long long most = std::min(2 * BATCH_SHAPES[shape].ppt, BATCH_TILE_MAX / 32);   // points a lane
    const long long k = std::max((m + lanes * most - 1) / (lanes * most), 1ll);
    return (int)(32 * std::min(std::max((m + lanes * k - 1) / (lanes * k), 1ll), most));
}

int batch_iter_blocks(int shape, BatchMode mode)
{
    if (shape < 0 || shape >= BATCH_N_SHAPES)
        return 0;
    IterKernel k = iter_kernel(shape, mode);
    const int threads = iter_threads(shape, mode);
    const size_t smem = iter_smem(threads);
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return sms * per_sm;
}

cudaError_t launch_batch_iter(int shape, BatchMode mode, int blocks, const BatchIterArgs &a, cudaStream_t st)
{
    IterKernel k = iter_kernel(shape, mode);
    if (!k || blocks < 1)
        return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(iter_threads(shape, mode));
    cfg.dynamicSmemBytes = iter_smem(iter_threads(shape, mode));
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, a);
}

}  // namespace vicp
