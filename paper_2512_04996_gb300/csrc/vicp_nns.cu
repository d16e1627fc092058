// vicp_nns.cu -- NNS (Alg. 4): localised search in the root voxel, and the
// global search for source points outside the grid or in unlabelled voxels.
#include "vicp_launch.h"
#include "vicp_search.cuh"

namespace vicp {

// ---------------------------------------------------------------------------
// Localised search: one thread per source point.  The point is transformed
// by the float-rounded pose, quantised, and its voxel's root label followed
// once (Alg. 4); the root voxel's CSR segment is scanned with 16-byte loads
// of (x, y, z, index), eight in flight.  A few dense voxels hold far more
// points than the rest, and a warp waits for its longest segment: a query
// whose segment has more than HEAVY points is not scanned here but listed,
// with its segment, for the next kernel, which gives each 4 to 32 lanes.
// Points that need the global search are listed for it.  Every list gets one
// global atomic per block.
// ---------------------------------------------------------------------------
constexpr int CORR_THREADS = 512;
// Whether a search of m points on grid g takes its near queries by rows of
// voxels (NEAR below).  Up to 16,384 points the global queries are so few that
// each has a warp of its own, and the brick search is as short a chain; and
// where a grid has many voxels for a query, few queries crowd round the same
// faces, and what the rows save does not pay for the longer code of both
// kernels, which is fetched cold in every iteration (the reduction's after it,
// too).  One search and update, grid kept, without / with: sphere and plane of
// 60,000 points (V = 17 m) 57.1 / 34.0 us, of 34,457 (V = m, 20 iterations)
// 1,381 / 984; an object of 40,000 (V = 50 m) 27.0 / 26.1; scenes (V = 48 m to
// 103 m) of 30,982 points 29.2 / 31.1, 60,000 31.2 / 33.5, 120,000 47.6 / 49.2.
constexpr int NEAR_MIN_QUERIES = 16384, NEAR_MAX_VOXELS = 32;

static bool near_by_rows(int m, const GridGeom &g)
{
    return m > NEAR_MIN_QUERIES && g.V <= (long long)NEAR_MAX_VOXELS * m;
}

// Segment of a root voxel in the CSR store: [off[r], off[r + 1]) (clamped to
// the store's length).
struct CsrSeg {
    const unsigned *off;
    unsigned cap;
    __device__ __forceinline__ void range(int r, unsigned &a, unsigned &b) const
    {
        a = __ldg(off + r);
        b = max(a, min(__ldg(off + r + 1), cap));
    }
};

// Segment of a root voxel in a fixed-capacity store: the first
// min(count[r], C) of the C slots that start at r * C.
struct FixedSeg {
    const unsigned *count;
    unsigned C;
    __device__ __forceinline__ void range(int r, unsigned &a, unsigned &b) const
    {
        a = (unsigned)r * C;
        b = a + min(__ldg(count + r), C);
    }
};

// Root label of voxel v, as the index of its segment in the store: the
// dense root array (the root's voxel key), or the sparse grid's two tables
// (the labelled-segment table gives v's row segment -- its label mask and
// the index of its first root -- and so the root's voxel key, at v's rank
// among the segment's labelled voxels; the occupied-voxel table gives that
// voxel's slot, which indexes the offsets).  -1: unlabelled.
struct DenseRoot {
    const int *root;
    __device__ __forceinline__ int operator()(int v) const { return __ldg(root + v); }
};

struct HashedRoot {
    const unsigned *lkeys;   // labelled row segments
    unsigned lmask;
    int lshift;
    const uint2 *lseg;       // their label masks and first-root indices
    const int *lroot;        // the labelled voxels' root keys, segment by segment
    const unsigned *okeys;   // occupied voxels
    unsigned omask;
    int oshift;
    int nx, nxb;             // grid row length, 32-voxel segments per row
    __device__ __forceinline__ int operator()(int v) const
    {
        const int x = v % nx, row = v / nx;   // row = y + ny z
        const int ls = hash_find(lkeys, lmask, lshift, (unsigned)((x >> 5) + nxb * row));
        if (ls < 0)
            return -1;
        const uint2 e = __ldg(lseg + ls);
        const unsigned bit = (unsigned)x & 31u;
        if (!((e.x >> bit) & 1u))
            return -1;
        const int r = __ldg(lroot + e.y + __popc(e.x & ((1u << bit) - 1u)));
        return hash_find(okeys, omask, oshift, (unsigned)r);
    }
};

template <bool NEAR, class Seg, class Root>
__global__ void __launch_bounds__(CORR_THREADS) k_correspond(const float4 *__restrict__ src, int m,
                                                             const double *__restrict__ pose, GridGeom g,
                                                             Root root, Seg seg,
                                                             const float4 *__restrict__ csr,
                                                             int *__restrict__ nn, float *__restrict__ d2,
                                                             int *__restrict__ fb_list, int *__restrict__ hv_list,
                                                             uint2 *__restrict__ hv_range, DevCtl *__restrict__ ctl,
                                                             int honor_stop)
{
    pdl_begin();
    if (honor_stop && *(volatile int *)&ctl->stop)
        return;
    __shared__ PoseF sp;
    __shared__ unsigned long long s_cand;   // block totals: one global atomic each
    __shared__ int s_fb, s_fb_base, s_nr, s_nr_base, s_hv, s_hv_base, s_no;
    if (threadIdx.x == 32) {   // (not the warp that loads the pose: the round trips overlap)
        s_cand = 0ull;
        s_fb = s_nr = s_hv = 0;
        s_no = NEAR ? __ldcg(&ctl->n_outside) : 0;
    }
    load_pose_f_block(pose, sp);   // also orders the initialisation above
    const PoseF P = sp;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    bool far = false, near = false, heavy = false;
    unsigned cand = 0u, a = 0u, b = 0u;
    if (i < m) {
        const float3 s = transform_pt(P, __ldg(src + i));
        bool inside = true;
        const int v = NEAR ? nearest_voxel(g, s, inside) : voxel_key(g, s.x, s.y, s.z);
        const int r = v >= 0 ? root(v) : -1;
        far = true;
        unsigned dense = 0u;
        if (r >= 0) {
            seg.range(r, a, b);
            dense = b - a;
            if (!inside)   // only a seed
                b = min(b, a + (unsigned)NEAR_SEED);
            cand = inside ? dense : 0u;
            heavy = cand > HEAVY;
            far = !inside;
        }
        if (NEAR ? !heavy : !heavy && !far) {   // (far without a label: an empty run, no seed)
            const unsigned long long best = segment_min(csr, a, b, s);
            nn[i] = (int)(unsigned)best;
            d2[i] = __uint_as_float((unsigned)(best >> 32));
            near = NEAR && far && dense && s_no <= NEAR_OUTSIDE_MAX &&
                   near_seed(s, __uint_as_float((unsigned)(best >> 32)), g.inv_h, dense);
            far = far && !near;
        }
    }
    const unsigned long long wc = warp_sum_u64(cand);
    unsigned fm = 0u, nm = 0u, hm = 0u;
    int fb_base = 0, nr_base = 0, hv_base = 0;
    const bool lists = __any_sync(FULL_MASK, far || near || heavy);
    if (lists) {
        fm = __ballot_sync(FULL_MASK, far);
        nm = __ballot_sync(FULL_MASK, near);
        hm = __ballot_sync(FULL_MASK, heavy);
    }
    if (lane == 0) {
        if (wc)
            atomicAdd(&s_cand, wc);
        if (fm)
            fb_base = atomicAdd(&s_fb, __popc(fm));
        if (nm)
            nr_base = atomicAdd(&s_nr, __popc(nm));
        if (hm)
            hv_base = atomicAdd(&s_hv, __popc(hm));
    }
    __syncthreads();
    // a thread of another warp for each counter: the round trips overlap
    if (threadIdx.x == 0 && s_fb)
        s_fb_base = atomicAdd(&ctl->fb_count, s_fb);
    if (threadIdx.x == 32 && s_nr)
        s_nr_base = atomicAdd(&ctl->nr_count, s_nr);
    if (threadIdx.x == 64 && s_hv)
        s_hv_base = atomicAdd(&ctl->hv_count, s_hv);
    if (threadIdx.x == 96) {
        if (s_cand)
            atomicAdd(&ctl->stat_local_cand, s_cand);
        if (blockIdx.x == 0)
            atomicAdd(&ctl->stat_queries, (unsigned long long)m);
    }
    __syncthreads();
    if (!lists)
        return;
    fb_base = __shfl_sync(FULL_MASK, fb_base, 0);
    nr_base = __shfl_sync(FULL_MASK, nr_base, 0);
    hv_base = __shfl_sync(FULL_MASK, hv_base, 0);
    if (near) {   // from the list's end: a query is in one of the two at most
        const int slot = s_nr_base + nr_base + __popc(nm & lanemask_lt());
        if (slot < m)
            fb_list[m - 1 - slot] = i;
        else
            atomicOr(&ctl->err, DEVERR_BOUNDS);
    }
    if (far) {
        const int slot = s_fb_base + fb_base + __popc(fm & lanemask_lt());
        if (slot < m)
            fb_list[slot] = i;
        else
            atomicOr(&ctl->err, DEVERR_BOUNDS);
    }
    if (heavy) {
        const int slot = s_hv_base + hv_base + __popc(hm & lanemask_lt());
        if (slot < m) {
            hv_list[slot] = i;
            hv_range[slot] = make_uint2(a, b);
        } else {
            atomicOr(&ctl->err, DEVERR_BOUNDS);
        }
    }
}

cudaError_t launch_correspond(const float4 *src, int m, const double *pose, const GridGeom &g, const int *root,
                              const unsigned *off, const float4 *csr, int n_cap, int *nn, float *d2,
                              int *fb_list, int *hv_list, uint2 *hv_range, DevCtl *ctl, int honor_stop,
                              cudaStream_t st)
{
    return launch_kernel(near_by_rows(m, g) ? k_correspond<true, CsrSeg, DenseRoot> : k_correspond<false, CsrSeg, DenseRoot>, dim3((m + CORR_THREADS - 1) / CORR_THREADS),
                         dim3(CORR_THREADS), 0, st, src, m, pose, g, DenseRoot{root}, CsrSeg{off, (unsigned)n_cap},
                         csr, nn, d2, fb_list, hv_list, hv_range, ctl, honor_stop);
}

cudaError_t launch_correspond_hashed(const float4 *src, int m, const double *pose, const GridGeom &g,
                                     const HashTable &labelled, const uint2 *lseg, const int *lroot,
                                     const HashTable &occupied, const unsigned *off, const float4 *csr, int n_cap,
                                     int *nn, float *d2, int *fb_list, int *hv_list, uint2 *hv_range, DevCtl *ctl,
                                     int honor_stop, cudaStream_t st)
{
    const HashedRoot root{labelled.keys, labelled.mask, labelled.shift, lseg, lroot,
                          occupied.keys, occupied.mask, occupied.shift, g.nx, (g.nx + 31) / 32};
    return launch_kernel(near_by_rows(m, g) ? k_correspond<true, CsrSeg, HashedRoot> : k_correspond<false, CsrSeg, HashedRoot>, dim3((m + CORR_THREADS - 1) / CORR_THREADS),
                         dim3(CORR_THREADS), 0, st, src, m, pose, g, root, CsrSeg{off, (unsigned)n_cap}, csr, nn, d2,
                         fb_list, hv_list, hv_range, ctl, honor_stop);
}

cudaError_t launch_correspond_fixed(const float4 *src, int m, const double *pose, const GridGeom &g, const int *root,
                                    const unsigned *count, unsigned C, const float4 *slots, int *nn, float *d2,
                                    int *fb_list, int *hv_list, uint2 *hv_range, DevCtl *ctl, cudaStream_t st)
{
    return launch_kernel(near_by_rows(m, g) ? k_correspond<true, FixedSeg, DenseRoot> : k_correspond<false, FixedSeg, DenseRoot>, dim3((m + CORR_THREADS - 1) / CORR_THREADS),
                         dim3(CORR_THREADS), 0, st, src, m, pose, g, DenseRoot{root}, FixedSeg{count, C}, slots, nn,
                         d2, fb_list, hv_list, hv_range, ctl, 0);
}

// ---------------------------------------------------------------------------
// Global search ("Globalsearch" of Alg. 4) of the queries the localised
// search listed (global_search: a warp per query over the brick levels), and
// the near queries (a group of 1 to 32 lanes each) and dense root segments
// (4 to 32) it listed.
//
// Scheduling without global atomics: block b takes the items b, b + B,
// b + 2B, ... of every list (B blocks; strided, so that a block's share
// mixes the regions of the source cloud and the shares cost about the
// same), far queries first, then a warp's worth of near queries or of dense
// segments at a time, and its warps take these items one at a time from a
// shared-memory counter.  Per-query
// costs vary several-fold, so the warps of a block balance each other; the
// shares balance the blocks.  (A single global ticket counter would put one
// same-address atomic per item, plus one per warp at the end, into the L2
// line that also holds the list lengths every block reads: on the 226k
// scene those ~17k serialised operations, not the searches, set the
// kernel's duration.)
// ---------------------------------------------------------------------------
constexpr int FB_THREADS = 256;

// Entries b, b + B, ... below n: how many (without a division while the
// blocks' shares are at most one).
__device__ __forceinline__ int strided_share(int n, int b, int B)
{
    return n <= b ? 0 : (n - b <= B ? 1 : (n - 1 - b) / B + 1);
}

template <bool NEAR, class Rows>
__global__ void __launch_bounds__(FB_THREADS, 4) k_fallback(const float4 *__restrict__ src,
                                                         const double *__restrict__ pose, GridGeom g, Rows rows,
                                                         const float4 *__restrict__ bpts,
                                                         const float4 *__restrict__ bbox,
                                                         const float4 *__restrict__ sb_box,
                                                         const float4 *__restrict__ tgt, int n_tgt,
                                                         const int *__restrict__ outside,
                                                         const int *__restrict__ fb_list,
                                                         const int *__restrict__ hv_list,
                                                         const uint2 *__restrict__ hv_range,
                                                         const float4 *__restrict__ csr,
                                                         DevCtl *__restrict__ ctl, int *__restrict__ nn,
                                                         float *__restrict__ d2, int m, int honor_stop,
                                                         int *__restrict__ n_global_out)
{
    pdl_begin();
    if (honor_stop && *(volatile int *)&ctl->stop)
        return;   // the correspond kernel appended nothing either
    __shared__ PoseF sp;
    __shared__ unsigned long long s_examined;   // block total: one global atomic
    __shared__ int s_n[5];                      // far, near, dense segments listed; super-bricks; targets outside
    __shared__ unsigned s_next;                 // next item of this block's share
    if (threadIdx.x >= 32 && threadIdx.x < 37) {   // (not the warp that loads the pose: the round trips overlap)
        const int k = threadIdx.x - 32;
        s_n[k] = __ldcg(k == 0 ? &ctl->fb_count : (k == 1 ? &ctl->nr_count : (k == 2 ? &ctl->hv_count :
                        (k == 3 ? &ctl->n_super : &ctl->n_outside))));
    }
    if (threadIdx.x == 64) {
        s_examined = 0ull;
        s_next = 0u;
    }
    load_pose_f_block(pose, sp);   // also orders the initialisation above
    const PoseF P = sp;
    const int lane = threadIdx.x & 31;
    const int F = min(s_n[0], m), N = NEAR ? min(s_n[1], m - F) : 0, Hv = min(s_n[2], m), ns = s_n[3], no = s_n[4];
    const int B = (int)gridDim.x, b = (int)blockIdx.x;
    // lanes a near query and a dense segment get (2^...), and how many of
    // them a warp takes at a time (2^...)
    const int gN = group_shift(N, B * FB_THREADS, NEAR_SHIFT_MIN), gH = group_shift(Hv, B * FB_THREADS, HEAVY_SHIFT_MIN);
    const int packN = 5 - gN, packH = 5 - gH;
    const int nG = strided_share(F, b, B), nN = strided_share((N + (1 << packN) - 1) >> packN, b, B),
              nH = strided_share((Hv + (1 << packH) - 1) >> packH, b, B);
    unsigned long long examined = 0ull;   // far queries: every lane counts the same; lane 0 reports
    unsigned examined_near = 0u;          // near queries: each lane its own

    for (;;) {
        int k = 0;
        if (lane == 0)
            k = (int)atomicAdd(&s_next, 1u);
        k = __shfl_sync(FULL_MASK, k, 0);
        if (k >= nG + nN + nH)
            break;
        if (k < nG) {   // a far query
            const int i = __ldg(fb_list + b + k * B);
            if ((unsigned)i >= (unsigned)m) {   // a stale entry: skip it, report it
                if (lane == 0)
                    atomicOr(&ctl->err, DEVERR_BOUNDS);
                continue;
            }
            const float3 s = transform_pt(P, __ldg(src + i));
            const unsigned long long best = global_search(s, bpts, bbox, sb_box, ns, tgt, n_tgt, outside, no, lane,
                                                          examined, NEAR ? nn_key(d2[i], nn[i]) : ~0ull);
            if (NEAR)
                __syncwarp();   // every lane has read the seed
            if (lane == 0) {
                nn[i] = (int)(unsigned)best;
                d2[i] = __uint_as_float((unsigned)(best >> 32));
            }
        } else if (NEAR && k < nG + nN) {   // near queries
            const int G = 1 << gN, q = ((b + (k - nG) * B) << packN) + (lane >> gN), sub = lane & (G - 1);
            const int i = q < N ? __ldg(fb_list + m - 1 - q) : -1;
            const bool on = (unsigned)i < (unsigned)m;
            if (!on && q < N)   // a stale entry: skip it, report it
                atomicOr(&ctl->err, DEVERR_BOUNDS);
            float3 s = make_float3(0.0f, 0.0f, 0.0f);
            unsigned long long best = ~0ull;
            if (on) {
                s = transform_pt(P, __ldg(src + i));
                best = nn_key(d2[i], nn[i]);
                for (int o = sub; o < no; o += G) {   // target points outside the grid
                    const int j = __ldg(outside + o);
                    best = umin64(best, nn_key(dist2(s, __ldg(tgt + j)), j));
                }
                examined_near += sub == 0 ? (unsigned)no : 0u;
            }
            if (no > 0)
                best = group_min(best, G);
            best = near_search(g, rows, s, best, on, sub, G, examined_near);
            if (on && sub == 0) {
                nn[i] = (int)(unsigned)best;
                d2[i] = __uint_as_float((unsigned)(best >> 32));
            }
        } else {        // dense root segments
            const int G = 1 << gH, q = ((b + (k - nG - nN) * B) << packH) + (lane >> gH), sub = lane & (G - 1);
            const int i = q < Hv ? __ldg(hv_list + q) : -1;
            const bool on = (unsigned)i < (unsigned)m;
            if (!on && q < Hv)
                atomicOr(&ctl->err, DEVERR_BOUNDS);
            unsigned long long best = ~0ull;
            if (on) {
                const uint2 r = __ldg(hv_range + q);
                best = group_scan(csr, r.x, r.y, transform_pt(P, __ldg(src + i)), sub, G);
            }
            best = group_min(best, G);
            if (on && sub == 0) {
                nn[i] = (int)(unsigned)best;
                d2[i] = __uint_as_float((unsigned)(best >> 32));
            }
        }
    }
    // work counter: one global atomic per block; the last block to finish
    // clears the list lengths for the next search
    examined = (lane == 0 ? examined : 0ull) + examined_near;
    examined = warp_sum_u64(examined);
    if (lane == 0 && examined)
        atomicAdd(&s_examined, examined);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_examined)
            atomicAdd(&ctl->stat_global_cand, s_examined);
        __threadfence();
        const unsigned done = atomicAdd(&ctl->fb_done, 1u);
        if (done == gridDim.x - 1) {
            ctl->stat_fallbacks += (unsigned long long)(F + N);
            if (n_global_out)
                *n_global_out = F + N;
            ctl->fb_count = 0;
            ctl->nr_count = 0;
            ctl->hv_count = 0;
            ctl->fb_done = 0u;
        }
    }
}

template <bool NEAR, class Rows>
static cudaError_t run_fallback(const FallbackArgs &a, const Rows &rows, cudaStream_t st)
{
    // as many warps as can be resident, and no more than there are queries
    static int per_sm = 0;
    if (per_sm == 0) {
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fallback<NEAR, Rows>, FB_THREADS, 0);
        if (e != cudaSuccess || per_sm < 1)
            per_sm = 1;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int blocks = min(sms * per_sm, (a.m + FB_THREADS / 32 - 1) / (FB_THREADS / 32));
    return launch_kernel(k_fallback<NEAR, Rows>, dim3(blocks), dim3(FB_THREADS), 0, st, a.src, a.pose, a.g, rows, a.bpts,
                         a.bbox, a.sb_box, a.tgt, a.n_tgt, a.outside, a.fb_list, a.hv_list, a.hv_range, a.hv_store,
                         a.ctl, a.nn, a.d2, a.m, a.honor_stop, a.n_global_out);
}

cudaError_t launch_fallback(const FallbackArgs &a, cudaStream_t st)
{
    if (!near_by_rows(a.m, a.g))   // no rows read
        return run_fallback<false>(a, CsrRows{a.occ, a.off, (unsigned)a.n_tgt, a.csr}, st);
    if (a.okeys.keys)
        return run_fallback<true>(a, HashedRows{a.occ, a.off, (unsigned)a.n_tgt, a.csr, a.okeys.keys, a.okeys.mask,
                                          a.okeys.shift}, st);
    return run_fallback<true>(a, CsrRows{a.occ, a.off, (unsigned)a.n_tgt, a.csr}, st);
}

}  // namespace vicp
