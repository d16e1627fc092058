// vicp_diff.cu -- the differentiable point-to-point loss of Eq. 1 over the
// pairs of a batch, and the se(3) maps its gradient needs.
//
// Loss of pair k at pose T with fixed correspondences nn (from the NNS of
// Alg. 4; they carry no gradient):
//     L_k = (1/M) sum_i |T p_i - q_nn(i)|^2.
// Its gradient under a left perturbation T <- Exp(d) T at d = 0, with
// d = (rho, phi) (translation part first):
//     dL/drho = (2/M) sum_i r_i,   dL/dphi = (2/M) sum_i s_i x r_i,
// s_i = T p_i, r_i = s_i - q_nn(i); and in a source point dL/dp_i =
// (2/M) R^T r_i.  For a pose parameterised as T = Exp(xi) T0 the gradient
// in xi is J(xi)^T times the left-perturbation gradient, J the left
// Jacobian of SE(3).
//
// s_i and r_i are formed in double-float arithmetic from the FP64 pose (the
// pose entries split into two floats), so the residual is exact to ~2^-48
// even where it is small against the coordinates; the sums are
// double-float, per item and then per pair in item order (deterministic).
#include <algorithm>

#include "vicp_batch.h"
#include "vicp_df.cuh"
#include "vicp_launch.h"

namespace vicp {

// ---------------------------------------------------------------------------
// SE(3) exponential and left Jacobian (FP64).  With
// t = |phi| and P = phi^ (the cross-product matrix):
//   Exp(rho, phi) = [[I + A P + B P^2, (I + B P + C P^2) rho], [0, 1]],
//   J(rho, phi)   = [[Js, Q], [0, Js]],  Js = I + B P + C P^2,
//   Q = R/2 + C (P R + R P + P R P) + D (P P R + R P P - 3 P R P)
//       + (D + 3 E)/2 (P R P P + P P R P),  R = rho^,
// with A = sin t / t, B = (1 - cos t)/t^2, C = (t - sin t)/t^3,
// D = (t^2/2 + cos t - 1)/t^4, E = (t - sin t - t^3/6)/t^5.  B is evaluated
// as 2 (sin(t/2)/t)^2; C, D and E lose digits to cancellation at small t, so
// for t < 2 they are summed from their Taylor series (terms
// (-1)^k t^2k / (2k + n)!, n = 3, 4, 5; E with the opposite sign).
//
// A warp per pose: lane 3i + j < 9 holds entry (i, j) of every 3x3 matrix, so
// that a product is three fused multiply-adds a lane on shuffled entries.
// (A thread per pose held all the matrices, and the series divided by their
// growing factors: a chain of some thousand FP64 operations on a pipe that
// takes a warp's operation 16 cycles: 64 poses 13.4 and 25.0 us for the
// exponential and the Jacobian.)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double m3_hat(int lane, double x, double y, double z)
{
    // [[0, -z, y], [z, 0, -x], [-y, x, 0]]
    return lane == 1 ? -z : (lane == 2 ? y : (lane == 3 ? z : (lane == 5 ? -x : (lane == 6 ? -y : (lane == 7 ? x : 0.0)))));
}

__device__ __forceinline__ double m3_mul(int lane, double a, double b)
{
    const int i = lane < 9 ? lane / 3 : 0, j = lane < 9 ? lane - 3 * i : 0;
    double c = __shfl_sync(FULL_MASK, a, 3 * i) * __shfl_sync(FULL_MASK, b, j);
    c = fma(__shfl_sync(FULL_MASK, a, 3 * i + 1), __shfl_sync(FULL_MASK, b, 3 + j), c);
    return fma(__shfl_sync(FULL_MASK, a, 3 * i + 2), __shfl_sync(FULL_MASK, b, 6 + j), c);
}

// Horner's scheme for sum over k of (-1)^k t2^k / (2k + N)!, t2 <= 4: fourteen
// terms (4^14 / 31! = 3e-26 is left out).
constexpr double factorial(int n) { return n < 2 ? 1.0 : (double)n * factorial(n - 1); }   // exact up to 22!

template <int N, int K>
__device__ __forceinline__ double taylor_tail(double t2)   // terms K and on, divided by (-t2)^K
{
    constexpr double c = 1.0 / factorial(2 * K + N);
    if constexpr (K == 13)
        return c;
    else
        return fma(-t2, taylor_tail<N, K + 1>(t2), c);
}

template <int N>
__device__ __forceinline__ double taylor_coeff(double t2)
{
    return taylor_tail<N, 0>(t2);
}

struct Se3Coeffs {
    double A, B, C, D, E;
};

__device__ inline Se3Coeffs se3_coeffs(double t)
{
    const double t2 = t * t;
    Se3Coeffs k;
    if (t < 1e-4) {
        k.A = 1.0 - t2 / 6.0 + t2 * t2 / 120.0;
        k.B = 0.5 - t2 / 24.0 + t2 * t2 / 720.0;
    } else {
        const double s = sin(0.5 * t) / t;
        k.A = sin(t) / t;
        k.B = 2.0 * s * s;
    }
    if (t < 2.0) {
        k.C = taylor_coeff<3>(t2);
        k.D = taylor_coeff<4>(t2);
        k.E = -taylor_coeff<5>(t2);
    } else {
        const double s = sin(t), c = cos(t);
        k.C = (t - s) / (t2 * t);
        k.D = (0.5 * t2 + c - 1.0) / (t2 * t2);
        k.E = (t - s - t2 * t / 6.0) / (t2 * t2 * t);
    }
    return k;
}

constexpr int SE3_WARPS = 4;   // poses per block

__global__ void __launch_bounds__(32 * SE3_WARPS) k_se3_exp(int n, const double *__restrict__ xi,
                                                            const double *__restrict__ T0, double *__restrict__ T)
{
    pdl_begin();
    const int k = blockIdx.x * SE3_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (k >= n)
        return;
    double x[6];
#pragma unroll
    for (int a = 0; a < 6; ++a)
        x[a] = xi[6 * (long long)k + a];
    // column c of T0, for lane 4a + c < 16
    const int a = (lane >> 2) & 3, c = lane & 3;
    double t0[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
        t0[r] = T0[16 * (long long)k + 4 * r + c];
    const double t = sqrt(x[3] * x[3] + x[4] * x[4] + x[5] * x[5]);
    const Se3Coeffs q = se3_coeffs(t);
    const double P = m3_hat(lane, x[3], x[4], x[5]);
    const double P2 = m3_mul(lane, P, P);
    const double I = lane == 0 || lane == 4 || lane == 8 ? 1.0 : 0.0;
    const double R = fma(q.B, P2, fma(q.A, P, I));
    const double J = fma(q.C, P2, fma(q.B, P, I));
    // row a of E = [R | J rho]
    const int r3 = a < 3 ? 3 * a : 0;
    const double e0 = __shfl_sync(FULL_MASK, R, r3), e1 = __shfl_sync(FULL_MASK, R, r3 + 1),
                 e2 = __shfl_sync(FULL_MASK, R, r3 + 2);
    double e3 = __shfl_sync(FULL_MASK, J, r3) * x[0];
    e3 = fma(__shfl_sync(FULL_MASK, J, r3 + 1), x[1], e3);
    e3 = fma(__shfl_sync(FULL_MASK, J, r3 + 2), x[2], e3);
    if (lane < 16)
        T[16 * (long long)k + lane] = a == 3 ? t0[3] : fma(e3, t0[3], fma(e2, t0[2], fma(e1, t0[1], e0 * t0[0])));
}

__global__ void __launch_bounds__(32 * SE3_WARPS) k_se3_jlt(int n, const double *__restrict__ xi,
                                                            const double *__restrict__ g, double *__restrict__ out)
{
    pdl_begin();
    const int k = blockIdx.x * SE3_WARPS + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (k >= n)
        return;
    double x[6], gk[6];
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        x[a] = xi[6 * (long long)k + a];
        gk[a] = g[6 * (long long)k + a];
    }
    const double t = sqrt(x[3] * x[3] + x[4] * x[4] + x[5] * x[5]);
    const Se3Coeffs c = se3_coeffs(t);
    const double P = m3_hat(lane, x[3], x[4], x[5]), Rh = m3_hat(lane, x[0], x[1], x[2]);
    const double P2 = m3_mul(lane, P, P), PR = m3_mul(lane, P, Rh), RP = m3_mul(lane, Rh, P);
    const double PRP = m3_mul(lane, PR, P), PPR = m3_mul(lane, P, PR), RPP = m3_mul(lane, RP, P);
    const double PRPP = m3_mul(lane, PRP, P), PPRP = m3_mul(lane, P, PRP);
    const double I = lane == 0 || lane == 4 || lane == 8 ? 1.0 : 0.0;
    const double Js = fma(c.C, P2, fma(c.B, P, I));
    const double Q = 0.5 * Rh + c.C * (PR + RP + PRP) + c.D * (PPR + RPP - 3.0 * PRP) +
                     0.5 * (c.D + 3.0 * c.E) * (PRPP + PPRP);
    // [[Js, Q], [0, Js]]^T g = (Js^T g_rho, Q^T g_rho + Js^T g_phi): entry j
    // on lane j < 3 and, of the second part, on lane 3 + j
    const int j = lane < 6 ? (lane < 3 ? lane : lane - 3) : 0;
    double js[3], qj[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        js[r] = __shfl_sync(FULL_MASK, Js, 3 * r + j);
        qj[r] = __shfl_sync(FULL_MASK, Q, 3 * r + j);
    }
    const double first = js[0] * gk[0] + js[1] * gk[1] + js[2] * gk[2];
    const double second = qj[0] * gk[0] + qj[1] * gk[1] + qj[2] * gk[2] + js[0] * gk[3] + js[1] * gk[4] + js[2] * gk[5];
    if (lane < 6)
        out[6 * (long long)k + lane] = lane < 3 ? first : second;
}

cudaError_t launch_se3_exp(int n, const double *xi, const double *T0, double *T, cudaStream_t st)
{
    return launch_kernel(k_se3_exp, dim3((n + SE3_WARPS - 1) / SE3_WARPS), dim3(32 * SE3_WARPS), 0, st, n, xi, T0, T);
}

cudaError_t launch_se3_jlt(int n, const double *xi, const double *g, double *out, cudaStream_t st)
{
    return launch_kernel(k_se3_jlt, dim3((n + SE3_WARPS - 1) / SE3_WARPS), dim3(32 * SE3_WARPS), 0, st, n, xi, g, out);
}

// ---------------------------------------------------------------------------
// The loss and its gradients: the (pair, tile) items are dealt out to the
// resident warps in contiguous shares.  A warp adds the sums [sum |r|^2,
// sum r, sum s x r] (the first alone when no pose gradient is asked for) over
// its items of one pair and leaves them in the first of those items' slots,
// zeros in the others; the warp that finishes a pair's last item adds the
// pair's slots in a fixed order and writes L_k and (if asked) dL_k * (2/M)
// (sum r, sum s x r).  Point gradients dL_k * (2/M) R^T r_i are written by the
// lane of the point.  Bound by the double-float arithmetic (some 350
// operations a point without the pose gradient, 500 with it).
// ---------------------------------------------------------------------------
constexpr int LOSS_THREADS = 256;
constexpr int LOSS_WARPS = LOSS_THREADS / 32;
constexpr int LOSS_SUMS = 7;
constexpr int LOSS_AHEAD = 2;   // points a lane loads before it works on them

__device__ __forceinline__ dfl df_of(double x)
{
    const float hi = __double2float_rn(x);
    return {hi, __double2float_rn(x - (double)hi)};
}

// (Three blocks an SM: left to itself the compiler takes 64 registers for the
// loss alone, and four, and 64 pairs of 20,000 points 41.6 us against 35.5.)
template <bool POSE_GRAD>
__global__ void __launch_bounds__(LOSS_THREADS, POSE_GRAD ? 0 : 3) k_batch_loss(const float4 *__restrict__ src,
                                                             const float4 *__restrict__ tgt,
                                                             const BatchPair *__restrict__ pairs,
                                                             BatchState *__restrict__ state,
                                                             const BatchItem *__restrict__ items, int n_items,
                                                             const double *__restrict__ pose,
                                                             const int *__restrict__ nn,
                                                             const double *__restrict__ dloss,
                                                             float2 *__restrict__ partials,
                                                             double *__restrict__ loss_out,
                                                             double *__restrict__ grad_pose,
                                                             float4 *__restrict__ grad_src, DevCtl *__restrict__ ctl,
                                                             unsigned *__restrict__ host_err)
{
    pdl_begin();
    constexpr int SUMS = POSE_GRAD ? LOSS_SUMS : 1;
    // A failed search (nobody has waited for it) has left nn as it was: no
    // number formed from it may look like a loss.  The status word also goes
    // to the host, whose next call of this context reports it.  (The kernel
    // itself sets DEVERR_MATCH alone, so every warp reads the same here.)
    const unsigned err = __ldcg(&ctl->err);
    const bool bad = (err & (DEVERR_TIMEOUT | DEVERR_BOUNDS)) != 0u;
    if ((err & ~DEVERR_DEGENERATE) && host_err && blockIdx.x == 0 && threadIdx.x == 0)
        *(volatile unsigned *)host_err = err;
    const float nan_f = __int_as_float(0x7fffffff);
    __shared__ dfl s_T[LOSS_WARPS][12];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long W = (long long)gridDim.x * LOSS_WARPS, gw = (long long)blockIdx.x * LOSS_WARPS + warp;
    const int x0 = (int)(gw * n_items / W), x1 = (int)((gw + 1) * n_items / W);
    dfl acc[SUMS];
    int first = x0;   // the first of this warp's items of the current pair
    for (int itx = x0; itx < x1; ++itx) {
        const BatchItem it = items[itx];
        const BatchPair *bp = pairs + it.pair;
        const int M = bp->n_src, tbase = bp->tbase, n_tgt = bp->n_tgt, n_own = bp->n_items;
        if (itx == x0 || itx == bp->item0) {   // a pair begins
            first = itx;
            __syncwarp();   // (the last pair's pose is no longer read)
            if (lane < 12)
                s_T[warp][lane] = df_of(pose[16 * it.pair + lane]);   // entry (a, b) of the 3x4 upper block at 4a + b
            __syncwarp();
#pragma unroll
            for (int k = 0; k < SUMS; ++k)
                acc[k] = {0.0f, 0.0f};
        }
        const dfl *T = s_T[warp];
        const double scale = bad ? (double)nan_f : 2.0 / (double)M * (dloss ? dloss[it.pair] : 1.0);
        const float scale_f = (float)scale;
#pragma unroll 1
        for (int i0 = it.i0 + lane; i0 < it.i1; i0 += 32 * LOSS_AHEAD) {
            // the loads of LOSS_AHEAD points first: the gather of a target
            // point waits for its index, and both come from memory
            int jj[LOSS_AHEAD];
            float4 pp[LOSS_AHEAD], qq[LOSS_AHEAD];
#pragma unroll
            for (int u = 0; u < LOSS_AHEAD; ++u) {
                jj[u] = -1;
                if (i0 + 32 * u < it.i1) {
                    jj[u] = __ldg(nn + i0 + 32 * u);
                    pp[u] = __ldg(src + i0 + 32 * u);
                }
            }
#pragma unroll
            for (int u = 0; u < LOSS_AHEAD; ++u) {
                if ((unsigned)jj[u] < (unsigned)n_tgt)
                    qq[u] = __ldg(tgt + tbase + jj[u]);
                else if (i0 + 32 * u < it.i1) {
                    if (bad) {
                        if (grad_src)
                            grad_src[i0 + 32 * u] = make_float4(nan_f, nan_f, nan_f, 0.0f);
                    } else {
                        atomicOr(&ctl->err, DEVERR_MATCH);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < LOSS_AHEAD; ++u) {
                if ((unsigned)jj[u] >= (unsigned)n_tgt)
                    continue;
                const int i = i0 + 32 * u;
                const float4 p = pp[u], q = qq[u];
                dfl s[3], r[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    dfl v = df_mul_f(T[4 * a], p.x);
                    v = df_add(v, df_mul_f(T[4 * a + 1], p.y));
                    v = df_add(v, df_mul_f(T[4 * a + 2], p.z));
                    s[a] = df_add(v, T[4 * a + 3]);
                    r[a] = df_sub(s[a], df_f(a == 0 ? q.x : (a == 1 ? q.y : q.z)));
                }
                acc[0] = df_acc(acc[0], df_add(df_add(df_mul(r[0], r[0]), df_mul(r[1], r[1])), df_mul(r[2], r[2])));
                if constexpr (POSE_GRAD) {
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        acc[1 + a] = df_acc(acc[1 + a], r[a]);
                    acc[4] = df_acc(acc[4], df_sub(df_mul(s[1], r[2]), df_mul(s[2], r[1])));
                    acc[5] = df_acc(acc[5], df_sub(df_mul(s[2], r[0]), df_mul(s[0], r[2])));
                    acc[6] = df_acc(acc[6], df_sub(df_mul(s[0], r[1]), df_mul(s[1], r[0])));
                }
                if (grad_src) {
                    // (2/M) dL R^T r, the residual rounded to float first (its
                    // double-float low part is below float resolution of the result)
                    const float rx = r[0].hi + r[0].lo, ry = r[1].hi + r[1].lo, rz = r[2].hi + r[2].lo;
                    float gv[3];
#pragma unroll
                    for (int b = 0; b < 3; ++b)   // (T's high parts are the entries rounded to float)
                        gv[b] = scale_f * (T[b].hi * rx + T[4 + b].hi * ry + T[8 + b].hi * rz);
                    grad_src[i] = make_float4(gv[0], gv[1], gv[2], 0.0f);
                }
            }
        }
        if (itx + 1 < x1 && itx + 1 < bp->item0 + n_own)   // the pair goes on in this warp
            continue;
        // the sums in a fixed order, the pair's when its last item is done
#pragma unroll
        for (int k = 0; k < SUMS; ++k) {
            dfl v = acc[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                v = df_add(v, df_shfl_xor(v, o));
            if (lane == k)
                partials[(size_t)first * LOSS_SUMS + k] = make_float2(v.hi, v.lo);
        }
        for (int z = first + 1; z <= itx; ++z)
            if (lane < SUMS)
                partials[(size_t)z * LOSS_SUMS + lane] = make_float2(0.0f, 0.0f);
        if (lane < SUMS)
            __threadfence();
        __syncwarp();
        unsigned last = 0u;
        if (lane == 0)
            last = atomicAdd(&state[it.pair].items_done, (unsigned)(itx - first + 1)) == (unsigned)(n_own - (itx - first + 1));
        if (!__shfl_sync(FULL_MASK, last, 0))
            continue;
        __threadfence();
        {   // lane k + 8 h adds sum k of items h, h + 4, ...
            const int k = lane & 7;
            const float2 *p0 = partials + (size_t)bp->item0 * LOSS_SUMS + k;
            dfl v = {0.0f, 0.0f};
            for (int b = lane >> 3; b < n_own; b += 32) {   // eight loads in flight
                float2 x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    x[u] = k < SUMS && b + 4 * u < n_own ? __ldcg(p0 + (size_t)(b + 4 * u) * LOSS_SUMS)
                                                         : make_float2(0.0f, 0.0f);
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    v = df_add(v, dfl{x[u].x, x[u].y});
            }
            v = df_add(v, df_shfl_xor(v, 8));
            v = df_add(v, df_shfl_xor(v, 16));
            const double sum = df_to_double(v);
            if (lane == 0)
                loss_out[it.pair] = bad ? (double)nan_f : sum / (double)M;
            else if (POSE_GRAD && lane < LOSS_SUMS && grad_pose)
                grad_pose[6 * it.pair + lane - 1] = scale * sum;
            if (lane == 0)
                state[it.pair].items_done = 0u;
        }
    }
}

template <bool POSE_GRAD>
static int loss_blocks()
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_loss<POSE_GRAD>, LOSS_THREADS, 0) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    return sms * per_sm;
}

cudaError_t launch_batch_loss(const float4 *src, const float4 *tgt, const BatchPair *pairs, BatchState *state,
                              const BatchItem *items, int n_items, const double *pose, const int *nn,
                              const double *dloss, float2 *partials, double *loss_out, double *grad_pose,
                              float4 *grad_src, DevCtl *ctl, unsigned *host_err, cudaStream_t st)
{
    static const int resident[2] = {loss_blocks<false>(), loss_blocks<true>()};
    const int blocks = std::min(resident[grad_pose != nullptr], (n_items + LOSS_WARPS - 1) / LOSS_WARPS);
    return launch_kernel(grad_pose ? k_batch_loss<true> : k_batch_loss<false>, dim3(blocks), dim3(LOSS_THREADS), 0, st,
                         src, tgt, pairs, state, items, n_items, pose, nn, dloss, partials, loss_out, grad_pose,
                         grad_src, ctl, host_err);
}

}  // namespace vicp
