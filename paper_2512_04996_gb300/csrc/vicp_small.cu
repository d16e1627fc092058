// vicp_small.cu -- ICP iterations of a small source cloud by one thread-block
// cluster: Alg. 4 and the update of Eq. 1, any number of iterations in one
// launch.
//
// A small cloud's iteration as three launches (localised search, global
// search, reduction and solve) is all latency: three launches, each with its
// own first loads, lists that go through global memory, a ticket for the last
// block and a solve whose code is fetched anew.  Here a cluster of up to 16
// blocks, a share of the points each, keeps the points' matches, the lists
// and the sums in shared memory for as many iterations as are asked for:
//   (1) thread per point: localised search (as k_correspond), queries without
//       a root and dense segments listed in shared memory;
//   (2) the block's warps answer its own lists: far queries a warp each,
//       near queries and dense segments 1 to 32 lanes each (as k_fallback);
//   (3) the block's sums in double-float, in a fixed order, written into the
//       shared memory of every block of the cluster; one cluster barrier (in
//       hardware, no polling);
//   (4) every block adds the blocks' sums in order and solves for itself, so
//       that no second barrier hands the pose out: all blocks compute the
//       same bits, and block 0 writes the results.
// Measured (30 iterations, grid kept, against the separate kernels): 4,096
// points 384-459 us against 709-753, 16,384 points 479-618 against 725-839
// (objects, by their share of global queries), 24,576 points (three a thread)
// 565-914 against 775-1,025; one step of 1,000 points 17.0 against 22.5.
// What bounds it now is the chain of an iteration: root, offset, points, the
// lists' rows, and the solve.  Past 24,576 points 16 SMs are too few for
// clouds with many global queries (40,960 points: an object 762 against 821,
// but a scene 1,497 against 952) and the separate kernels serve.
// The sums are bit-reproducible from run to run, and k_reduce_solve adds those
// of a small cloud in the same order, so that an iteration by the separate
// kernels gives the same bits.  The slots of two
// iterations alternate: a block overwrites a slot only after the barrier
// that every reader of it has passed.
#include <mutex>

#include "vicp_df.cuh"
#include "vicp_launch.h"
#include "vicp_search.cuh"

namespace vicp {

constexpr int SM_THREADS = SMALL_THREADS, SM_WARPS = SM_THREADS / 32;
constexpr int SM_CLUSTER = SMALL_CLUSTER;
constexpr int SM_PPT_MAX = SMALL_MAX_POINTS / (SM_CLUSTER * SM_THREADS);   // points per thread, at most
static_assert(SM_PPT_MAX * SM_CLUSTER * SM_THREADS == SMALL_MAX_POINTS, "points per thread");
constexpr size_t SM_SMEM = (size_t)2 * SM_WARPS * N_SUMS * 33 * sizeof(float);   // transposed per-lane sums

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Stores v at the address that p has in block `rank` of the cluster.
__device__ __forceinline__ void store_remote(dfl *p, unsigned rank, dfl v)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(r), "f"(v.hi), "f"(v.lo) : "memory");
}

template <int SM_PPT>
__global__ void __launch_bounds__(SM_THREADS, 1) k_small_iters(const SmallArgs a)
{
    constexpr int SM_POINTS = SM_THREADS * SM_PPT;   // points per block
    pdl_begin();
    if (a.honor_stop && *(volatile int *)&a.ctl->stop)   // (the same for every block)
        return;
    __shared__ double s_pose[16];
    __shared__ PoseF s_P;
    __shared__ unsigned long long s_key[SM_POINTS];   // each point's best key; the seed while it is listed
    __shared__ short s_list[SM_POINTS];               // far queries from the front, near ones from the back
    __shared__ short s_hv[SM_POINTS];                 // dense segments
    __shared__ uint2 s_range[SM_POINTS];              // ... their runs, by point
    __shared__ int s_far, s_near, s_heavy, s_stop;
    __shared__ float s_hi[SM_WARPS][N_SUMS], s_lo[SM_WARPS][N_SUMS];
    __shared__ dfl s_part[2][SM_CLUSTER][N_SUMS];     // the blocks' sums of two iterations
    __shared__ dfl s_tot[N_SUMS];
    extern __shared__ float s_dyn[];
    float(*s_thi)[N_SUMS][33] = reinterpret_cast<float(*)[N_SUMS][33]>(s_dyn);
    float(*s_tlo)[N_SUMS][33] = reinterpret_cast<float(*)[N_SUMS][33]>(s_dyn + SM_WARPS * N_SUMS * 33);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned rank = cluster_rank();
    const int blocks = (int)gridDim.x;   // one cluster
    const GridGeom &g = a.g;
    const CsrRows rows{a.occ, a.off, (unsigned)a.n_tgt, a.csr};
    const int ns = __ldcg(&a.ctl->n_super), no = __ldcg(&a.ctl->n_outside);
    // the loop so far (read before the first barrier; block 0 writes it at the end)
    const int it0 = a.honor_stop ? *(volatile int *)&a.ctl->iters : 0;
    double prev = a.honor_stop ? *(volatile double *)&a.ctl->prev_rmse : 0.0;
    if (tid < 16)
        s_pose[tid] = a.pose[tid];

    // this thread's points: tiles of 32 dealt out to the blocks in turn, so
    // that every block gets a mix of the cloud's regions
    float4 p[SM_PPT];
#pragma unroll
    for (int u = 0; u < SM_PPT; ++u) {
        const int l = tid + SM_THREADS * u, i = ((l >> 5) * blocks + (int)rank) * 32 + lane;
        p[u] = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(i < a.m ? 1 : 0));
        if (i < a.m) {
            const float4 q = __ldg(a.src + i);
            p[u].x = q.x;
            p[u].y = q.y;
            p[u].z = q.z;
        }
    }
    unsigned long long st_cand = 0ull, st_glob = 0ull, st_far = 0ull;   // work counters
    unsigned near_cand = 0u;
    cluster_barrier();   // every block has started: its shared memory may be written
    int done = 0;
    double rmse = 0.0;
    bool ok = true;
    for (int it = 0; it < a.iters; ++it) {
        if (tid < 12) {
            const int r = tid >> 2, c = tid & 3;
            const float v = __double2float_rn(s_pose[tid]);
            if (c < 3)
                s_P.r[3 * r + c] = v;
            else
                s_P.t[r] = v;
        }
        if (tid == 32)
            s_far = s_near = s_heavy = 0;
        __syncthreads();
        const PoseF P = s_P;

        // (1) localised search
        float3 s[SM_PPT];
#pragma unroll
        for (int u = 0; u < SM_PPT; ++u) {
            s[u] = transform_pt(P, p[u]);
            if (__float_as_int(p[u].w) == 0)
                continue;
            const int l = tid + SM_THREADS * u;
            bool inside;
            const int v = nearest_voxel(g, s[u], inside);
            const int r = v >= 0 ? __ldg(a.root + v) : -1;
            unsigned x0 = 0u, x1 = 0u, dense = 0u;
            if (r >= 0) {
                x0 = __ldg(rows.off + r);
                x1 = max(x0, min(__ldg(rows.off + r + 1), rows.cap));
                dense = x1 - x0;
                if (!inside)   // only a seed
                    x1 = min(x1, x0 + (unsigned)NEAR_SEED);
            }
            if (inside && r >= 0) {
                st_cand += dense;
                if (dense > HEAVY) {
                    s_hv[atomicAdd(&s_heavy, 1)] = (short)l;
                    s_range[l] = make_uint2(x0, x1);
                    continue;
                }
            }
            const unsigned long long best = segment_min(rows.csr, x0, x1, s[u]);
            s_key[l] = best;
            if (!(inside && r >= 0)) {
                if (dense && no <= NEAR_OUTSIDE_MAX && near_seed(s[u], __uint_as_float((unsigned)(best >> 32)), g.inv_h, dense))
                    s_list[SM_POINTS - 1 - atomicAdd(&s_near, 1)] = (short)l;
                else
                    s_list[atomicAdd(&s_far, 1)] = (short)l;
            }
        }
        __syncthreads();

        // (2) the block's lists (the order within a list varies, a query's
        //     answer does not)
        const int F = s_far, N = s_near, Hv = s_heavy;
        auto point_of = [&](int l) {
            const int i = ((l >> 5) * blocks + (int)rank) * 32 + (l & 31);
            return transform_pt(P, __ldg(a.src + i));
        };
        for (int k = warp; k < F; k += SM_WARPS) {
            const int l = s_list[k];
            const unsigned long long best = global_search(point_of(l), a.bpts, a.bbox, a.sb_box, ns, a.tgt, a.n_tgt,
                                                          a.outside, no, lane, st_glob, s_key[l]);
            __syncwarp();
            if (lane == 0)
                s_key[l] = best;
        }
        {
            const int shift = group_shift(N, SM_THREADS, NEAR_SHIFT_MIN), G = 1 << shift, pack = 32 >> shift;
            const int sub = lane & (G - 1);
            for (int k = (SM_WARPS - 1 - warp) * pack; k < N; k += SM_WARPS * pack) {
                const int q = k + (lane >> shift);
                const bool on = q < N;
                const int l = on ? s_list[SM_POINTS - 1 - q] : 0;
                float3 t = make_float3(0.0f, 0.0f, 0.0f);
                unsigned long long best = ~0ull;
                if (on) {
                    t = point_of(l);
                    best = s_key[l];
                    for (int o = sub; o < no; o += G) {   // target points outside the grid
                        const int j = __ldg(a.outside + o);
                        best = umin64(best, nn_key(dist2(t, __ldg(a.tgt + j)), j));
                    }
                    near_cand += sub == 0 ? (unsigned)no : 0u;
                }
                best = group_min(best, G);
                best = near_search(g, rows, t, best, on, sub, G, near_cand);
                if (on && sub == 0)
                    s_key[l] = best;
            }
        }
        {
            const int shift = group_shift(Hv, SM_THREADS, HEAVY_SHIFT_MIN), G = 1 << shift, pack = 32 >> shift;
            const int sub = lane & (G - 1);
            for (int k = warp * pack; k < Hv; k += SM_WARPS * pack) {
                const int q = k + (lane >> shift);
                const int l = q < Hv ? s_hv[q] : -1;
                unsigned long long best = ~0ull;
                if (l >= 0) {
                    const uint2 r = s_range[l];
                    best = group_scan(rows.csr, r.x, r.y, point_of(l), sub, G);
                }
                best = group_min(best, G);
                if (l >= 0 && sub == 0)
                    s_key[l] = best;
            }
        }
        if (tid == 0)
            st_far += (unsigned long long)(F + N);
        __syncthreads();

        // (3) the block's sums: thread, warp (through shared memory, as
        //     k_reduce_solve), block
        dfl acc[N_SUMS];
#pragma unroll
        for (int k = 0; k < N_SUMS; ++k)
            acc[k] = {0.0f, 0.0f};
#pragma unroll
        for (int u = 0; u < SM_PPT; ++u) {
            if (__float_as_int(p[u].w) == 0)
                continue;
            const int j = (int)(unsigned)s_key[tid + SM_THREADS * u];
            if ((unsigned)j < (unsigned)a.n_tgt)
                accumulate_corr(acc, s[u], __ldg(a.tgt + j), a.center);
            else   // no valid match: report, leave it out
                atomicOr(&a.ctl->err, DEVERR_BOUNDS);
        }
#pragma unroll
        for (int k = 0; k < N_SUMS; ++k) {
            s_thi[warp][k][lane] = acc[k].hi;
            s_tlo[warp][k][lane] = acc[k].lo;
        }
        __syncwarp();
        {
            const int k = lane & 15, h = (lane >> 4) * 16;
            dfl v = {s_thi[warp][k][h], s_tlo[warp][k][h]};
#pragma unroll
            for (int t = 1; t < 16; ++t)
                v = df_acc(v, dfl{s_thi[warp][k][h + t], s_tlo[warp][k][h + t]});
            v = df_acc(v, df_shfl_xor(v, 16));
            if (lane < 16) {
                s_hi[warp][k] = v.hi;
                s_lo[warp][k] = v.lo;
            }
        }
        __syncthreads();
        dfl(*part)[N_SUMS] = s_part[it & 1];
        if (warp == 0) {   // the block's warps in order (the halves of the warp half of them each)
            const int k = lane & 15, w0 = (lane >> 4) * (SM_WARPS / 2);
            dfl v = {s_hi[w0][k], s_lo[w0][k]};
#pragma unroll
            for (int w = 1; w < SM_WARPS / 2; ++w)
                v = df_acc(v, dfl{s_hi[w0 + w][k], s_lo[w0 + w][k]});
            v = df_acc(v, df_shfl_xor(v, 16));
            for (int c = lane >> 4; c < blocks; c += 2)   // two blocks' slots at a time
                store_remote(&part[rank][k], (unsigned)c, v);
            __syncwarp();
        }
        cluster_barrier();

        // (4) the blocks' sums in order, and the solve
        if (warp == 0) {
            const int k = lane & 15, half = (blocks + 1) / 2, c0 = (lane >> 4) * half, c1 = min(c0 + half, blocks);
            dfl v = {0.0f, 0.0f};
            for (int c = c0; c < c1; ++c)
                v = df_acc(v, part[c][k]);
            v = df_acc(v, df_shfl_xor(v, 16));
            if (lane < 16)
                s_tot[k] = v;
            __syncwarp();
            ok = solve_update(s_tot, a.m, a.center, s_pose, rmse);
            const bool converged = a.honor_stop && ok && a.eps > 0.0 && it0 + it >= 1 && fabs(rmse - prev) < a.eps;
            prev = rmse;
            if (lane == 0)
                s_stop = !ok || converged;
            done += ok ? 1 : 0;
        }
        __syncthreads();
        if (s_stop)   // the same in every block: they solved the same sums
            break;
    }

    if (rank == 0 && warp == 0) {
        if (lane < 12)
            a.pose[lane] = s_pose[lane];
        if (lane == 0) {
            if (a.rmse_out)
                *a.rmse_out = rmse;
            if (!ok)
                atomicOr(&a.ctl->err, DEVERR_DEGENERATE);
            if (a.honor_stop) {
                a.ctl->stop = s_stop;
                a.ctl->iters = it0 + done;
                a.ctl->last_rmse = rmse;
                a.ctl->prev_rmse = rmse;
            }
            atomicAdd(&a.ctl->stat_queries, (unsigned long long)a.m * (unsigned long long)(done + (ok ? 0 : 1)));
        }
    }
    st_glob = (lane == 0 ? st_glob : 0ull) + near_cand;
    st_cand = warp_sum_u64(st_cand);
    st_glob = warp_sum_u64(st_glob);
    if (lane == 0) {
        if (st_cand)
            atomicAdd(&a.ctl->stat_local_cand, st_cand);
        if (st_glob)
            atomicAdd(&a.ctl->stat_global_cand, st_glob);
        if (st_far)
            atomicAdd(&a.ctl->stat_fallbacks, st_far);
    }
}

using SmallKernel = void (*)(const SmallArgs);

// Points per thread for m points: as few as a full cluster needs.
static SmallKernel small_kernel(int m)
{
    constexpr int per = SM_CLUSTER * SM_THREADS;
    return m <= per ? k_small_iters<1> : (m <= 2 * per ? k_small_iters<2> : k_small_iters<SM_PPT_MAX>);
}

static cudaLaunchConfig_t small_config(int blocks, cudaLaunchAttribute (&attr)[2], cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(SM_THREADS);
    cfg.dynamicSmemBytes = SM_SMEM;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

// A cluster of 16 is past the portable size and needs a device with that many
// free SMs in one processing cluster: where it cannot be had, the separate
// kernels serve.
static bool small_iters_fit()
{
    for (int m : {1, 2 * SM_CLUSTER * SM_THREADS, SMALL_MAX_POINTS}) {
        const SmallKernel k = small_kernel(m);
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = small_config(SM_CLUSTER, attr, nullptr);
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM_SMEM) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess || n < 1) {
            cudaGetLastError();
            return false;
        }
    }
    return true;
}

// The answer is the device's: asked once for each, by the first call that
// wants it (it loads the kernels: the first context of a process took 1.08 ms
// to create with it and takes 0.55 without, also where none ever needs them).
bool small_iters_usable(int device)
{
    constexpr int MAX_DEVICES = 64;
    static std::mutex lock;
    static signed char known[MAX_DEVICES];   // 0: not asked; 1: yes; -1: no
    if (device < 0 || device >= MAX_DEVICES)
        return false;
    std::lock_guard<std::mutex> hold(lock);
    if (known[device] == 0)
        known[device] = small_iters_fit() ? 1 : -1;
    return known[device] > 0;
}

cudaError_t launch_small_iters(const SmallArgs &a, cudaStream_t st)
{
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = small_config(small_blocks(a.m), attr, st);
    return cudaLaunchKernelEx(&cfg, small_kernel(a.m), a);
}

}  // namespace vicp
