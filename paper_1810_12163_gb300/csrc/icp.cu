// ICP of a camera pose against the scene model before ranking (Sec. 3.2.4).
// The paper refines each chosen pose by ICP and drops the pose when ICP
// fails; the ICP variant is its host system's.  Here: point-to-plane ICP
// against the analytic room box with projective association, Gauss-Newton
// on a camera-frame update H exp(xi), coarse to fine over pixel strides (the
// rules are stated with rl_icp_params in the public header).
//
// One thread block owns one (frame, pose) for all iterations: its threads
// stride over the level's pixels accumulating the normal equations in FP32
// registers, the sums are reduced across lanes by shuffles and across warps
// in warp order in FP64, and one thread solves the ridged 6x6 system in FP64
// and composes the update.  The frame's depth image stays in L2 across the
// poses and iterations that read it.
//
// The camera-frame Jacobian J = (m, x x m), m = R^T n, equals B J_w with
// B = diag(R^T, R^T) and the world-frame J_w = (n, q' x n), q' = R x = d dir.
// With n = e_a a face axis, J_w has three nonzero entries, so each pixel adds
// 9 terms to the sums of its face axis (27 in all) instead of 27 terms of a
// dense J.  B is orthogonal: the ridged system is solved in the world frame
// (same trace, same ridge) and the step is rotated back, xi = B xi_w.
#include <cooperative_groups.h>

#include <type_traits>

#include "kernels.h"
#include "lm_dev.cuh"

namespace rl {

constexpr int ICP_THREADS = 256;
constexpr int ICP_WARPS = ICP_THREADS / 32;
// Sums per face axis a (i1 = a+1, i2 = a+2 mod 3; the rotational entries of
// J_w are P1 = q'[i2] at w[i1] and P2 = -q'[i1] at w[i2]): count, P1, P2,
// P1^2, P2^2, P1 P2, r, P1 r, P2 r.
constexpr int ICP_NS = 27;

template <int O>
__device__ __forceinline__ void icp_add(float acc[ICP_NS], float P1, float P2, float r) {
    acc[O] += 1.f;
    acc[O + 1] = __fadd_rn(acc[O + 1], P1);
    acc[O + 2] = __fadd_rn(acc[O + 2], P2);
    acc[O + 3] = fmaf(P1, P1, acc[O + 3]);
    acc[O + 4] = fmaf(P2, P2, acc[O + 4]);
    acc[O + 5] = fmaf(P1, P2, acc[O + 5]);
    acc[O + 6] = __fadd_rn(acc[O + 6], r);
    acc[O + 7] = fmaf(P1, r, acc[O + 7]);
    acc[O + 8] = fmaf(P2, r, acc[O + 8]);
}

// One live pixel (u, v) with depth d against the pose (R, t): its ray
// direction in the world and the signed gap to the model point along it, when
// there is one within sqrt(dist2); returns the hit face's axis, or -1.
// INSIDE: the camera centre lies strictly inside the box (known per pose), so
// the first face hit is the exit face, s = min over axes of the distance to
// the face the ray heads for; otherwise the general slab test (exit from
// inside, entry from outside).  exit_num[ax] = (hi - t, t - lo) for the two
// ray directions.  Here and in the sums, products and additions that the
// compiler may or may not fuse are rounded by name: the kernels below have to
// agree to the bit whatever it would make of each of them.
template <bool INSIDE>
__device__ __forceinline__ int icp_gap(const IcpArgs &a, float d, int u, int v, float cx, float cy, float ifx,
                                       float ify, const float R[9], const float t[3], const float exit_hi[3],
                                       const float exit_lo[3], float dist2, float dir[3], float &gap, int &n_valid) {
    if (!(d > 0.f) || isinf(d)) return -1;
    ++n_valid;
    const float c0 = ((float)u - cx) * ifx, c1 = ((float)v - cy) * ify;
#pragma unroll
    for (int r = 0; r < 3; ++r) dir[r] = fmaf(R[3 * r], c0, fmaf(R[3 * r + 1], c1, R[3 * r + 2]));
    int ax;
    if (INSIDE) {
        // exit distance along axis k: e_k / |dir_k| (e_k > 0); the smallest is
        // found by cross-multiplication (a zero |dir_k| never wins), then one
        // division
        float na = dir[0] > 0.f ? exit_hi[0] : exit_lo[0], da = fabsf(dir[0]);
        ax = 0;
#pragma unroll
        for (int k = 1; k < 3; ++k) {
            const float nk = dir[k] > 0.f ? exit_hi[k] : exit_lo[k], dk = fabsf(dir[k]);
            if (nk * da < na * dk) { na = nk; da = dk; ax = k; }
        }
        gap = fmaf(-na, rcp_approx(da), d);
    } else {
        float tn = -INFINITY, tf = INFINITY;
        int an = 0, af = 0;
        bool hit = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (dir[k] == 0.f) {
                hit = hit && t[k] >= a.lo[k] && t[k] <= a.hi[k];
                continue;
            }
            const float inv = rcp_approx(dir[k]);
            const float t1 = __fmul_rn(a.lo[k] - t[k], inv), t2 = __fmul_rn(a.hi[k] - t[k], inv);
            const float tmin = fminf(t1, t2), tmax = fmaxf(t1, t2);
            if (tmin > tn) { tn = tmin; an = k; }
            if (tmax < tf) { tf = tmax; af = k; }
        }
        if (!hit || tn > tf || !(tf > 0.f)) return -1;
        gap = __fsub_rn(d, tn > 0.f ? tn : tf);
        ax = tn > 0.f ? an : af;
    }
    const float dd2 = fmaf(dir[0], dir[0], fmaf(dir[1], dir[1], dir[2] * dir[2]));
    return gap * gap * dd2 > dist2 ? -1 : ax;
}

// Adds the point-to-plane terms of a pixel whose model point lies on a face
// of axis ax.
__device__ __forceinline__ void icp_terms(int ax, float d, float gap, float dir0, float dir1, float dir2,
                                          float acc[ICP_NS]) {
    // q' = d dir (the camera point rotated into the world frame); residual
    // r = n . (q - p) = gap dir[ax]
    const float q0 = __fmul_rn(d, dir0), q1 = __fmul_rn(d, dir1), q2 = __fmul_rn(d, dir2);
    // neighbouring pixels of a warp mostly share a face, so the branch on
    // the axis rarely diverges; constant offsets keep acc in registers
    if (ax == 0)
        icp_add<0>(acc, q2, -q1, __fmul_rn(gap, dir0));
    else if (ax == 1)
        icp_add<9>(acc, q0, -q2, __fmul_rn(gap, dir1));
    else
        icp_add<18>(acc, q1, -q0, __fmul_rn(gap, dir2));
}

// The same for the sums of one axis, given q' there (P1, P2) and the residual;
// zeros leave the sums as they are.
__device__ __forceinline__ void icp_add_axis(float s[9], bool on, float P1, float P2, float r) {
    const float u = on ? P1 : 0.f, v = on ? P2 : 0.f, w = on ? r : 0.f;
    s[0] += on ? 1.f : 0.f;
    s[1] = __fadd_rn(s[1], u);
    s[2] = __fadd_rn(s[2], v);
    s[3] = fmaf(u, u, s[3]);
    s[4] = fmaf(v, v, s[4]);
    s[5] = fmaf(u, v, s[5]);
    s[6] = __fadd_rn(s[6], w);
    s[7] = fmaf(u, w, s[7]);
    s[8] = fmaf(v, w, s[8]);
}

template <bool INSIDE>
__device__ __forceinline__ void icp_pixel(const IcpArgs &a, float d, int u, int v, float cx, float cy, float ifx,
                                          float ify, const float R[9], const float t[3], const float exit_hi[3],
                                          const float exit_lo[3], float dist2, float acc[ICP_NS], int &n_in,
                                          int &n_valid) {
    float dir[3], gap;
    const int ax = icp_gap<INSIDE>(a, d, u, v, cx, cy, ifx, ify, R, t, exit_hi, exit_lo, dist2, dir, gap, n_valid);
    if (ax < 0) return;
    icp_terms(ax, d, gap, dir[0], dir[1], dir[2], acc);
    ++n_in;
}

// The thread's pixels of one level: grid cells (iu, iv) ICP_THREADS apart
// in row-major order, stepped without divisions; ICP_LOADS depths are loaded
// before any is used, so that their latencies overlap.
constexpr int ICP_LOADS = 4;

template <bool INSIDE>
__device__ __forceinline__ void icp_sweep(const Frame &fr, const IcpArgs &a, int iu, int iv, int du, int dv, int nu,
                                          int nv, int st, float ifx, float ify, const float R[9], const float t[3],
                                          const float exit_hi[3], const float exit_lo[3], float dist2,
                                          float acc[ICP_NS], int &n_in, int &n_valid) {
    while (iv < nv) {
        float dk[ICP_LOADS];
        int uk[ICP_LOADS], vk[ICP_LOADS];
#pragma unroll
        for (int j = 0; j < ICP_LOADS; ++j) {
            uk[j] = iu * st;
            vk[j] = iv * st;
            dk[j] = iv < nv ? fr.depth[(size_t)vk[j] * fr.W + uk[j]] : 0.f;  // 0: no pixel
            iu += du;
            iv += dv;
            if (iu >= nu) {
                iu -= nu;
                ++iv;
            }
        }
#pragma unroll
        for (int j = 0; j < ICP_LOADS; ++j)
            icp_pixel<INSIDE>(a, dk[j], uk[j], vk[j], fr.cx, fr.cy, ifx, ify, R, t, exit_hi, exit_lo, dist2, acc,
                              n_in, n_valid);
    }
}

// One Gauss-Newton step from the reduced per-axis sums (thread 0 only; kept
// out of line so that its FP64 temporaries do not raise the pixel loop's
// register count): assembles the world-frame system, solves (A_w + lambda I)
// xi_w = -g_w with lambda = ridge * trace / 6, rotates the step into the
// camera frame and sets H <- H exp(xi).  False when there are fewer than 6
// inliers or the system is not positive definite.
__device__ __noinline__ bool icp_step(double *sH, const double *s_tot, double ridge) {
    double A[36], g[6], xi[6];
    for (int k = 0; k < 36; ++k) A[k] = 0.0;
    for (int k = 0; k < 6; ++k) g[k] = 0.0;
    double n_in = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double *S = s_tot + 9 * a;
        const int w1 = 3 + (a + 1) % 3, w2 = 3 + (a + 2) % 3;
        n_in += S[0];
        A[7 * a] += S[0];
        A[6 * a + w1] += S[1]; A[6 * w1 + a] += S[1];
        A[6 * a + w2] += S[2]; A[6 * w2 + a] += S[2];
        A[7 * w1] += S[3];
        A[7 * w2] += S[4];
        A[6 * w1 + w2] += S[5]; A[6 * w2 + w1] += S[5];
        g[a] -= S[6];
        g[w1] -= S[7];
        g[w2] -= S[8];
    }
    if (n_in < 6.0) return false;
    const double lam = ridge * (A[0] + A[7] + A[14] + A[21] + A[28] + A[35]) / 6.0;
    for (int r = 0; r < 6; ++r) A[7 * r] += lam;
    double xw[6];
    if (!chol_solve6(A, g, xw)) return false;
    // xi = diag(R^T, R^T) xi_w
    for (int r = 0; r < 3; ++r) {
        xi[r] = sH[r] * xw[0] + sH[4 + r] * xw[1] + sH[8 + r] * xw[2];
        xi[3 + r] = sH[r] * xw[3] + sH[4 + r] * xw[4] + sH[8 + r] * xw[5];
    }
    // H <- H exp(xi): exp(xi) as the left update of the identity
    double E[12] = {1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0}, N[12];
    se3_left(xi, E);
    for (int r = 0; r < 3; ++r)
        for (int q = 0; q < 4; ++q)
            N[4 * r + q] = sH[4 * r] * E[q] + sH[4 * r + 1] * E[4 + q] + sH[4 * r + 2] * E[8 + q] +
                           (q == 3 ? sH[4 * r + 3] : 0.0);
    for (int q = 0; q < 12; ++q) sH[q] = N[q];
    return true;
}

__global__ void __launch_bounds__(ICP_THREADS, 3) k_icp(IcpArgs a) {
    const int b = blockIdx.y, c = blockIdx.x;
    if (a.gate && a.gate[b] <= 0) return;
    const int cnt = a.counts ? a.counts[b] : a.cap;
    if (c >= cnt) return;
    const Frame fr = a.frames[b];
    double *P = a.poses + ((size_t)b * a.pose_stride + c) * 12;
    __shared__ double sH[12];
    __shared__ float s_part[ICP_WARPS][ICP_NS];
    __shared__ int s_cnt[ICP_WARPS][2];
    __shared__ double s_tot[ICP_NS];
    __shared__ int s_n[2];  // inliers, valid pixels of the last iteration
    __shared__ int s_fail;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid < 12) sH[tid] = P[tid];
    if (tid == 0) {
        s_fail = 0;
        s_n[0] = s_n[1] = 0;
    }
    const float ifx = 1.0f / fr.fx, ify = 1.0f / fr.fy;
    unsigned long long visited = 0;
    bool stop = false;
    for (int l = 0; l < a.ip.levels && !stop; ++l) {
        const int st = a.ip.stride[l];
        const int nu = (fr.W + st - 1) / st, nv = (fr.H + st - 1) / st;
        const float dist2 = a.ip.dist[l] * a.ip.dist[l];
        // the level's pixels (column iu, row iv of the strided grid) visited
        // ICP_THREADS apart in row-major order, stepped without divisions
        const int du = nu > 0 ? ICP_THREADS % nu : 0, dv = nu > 0 ? ICP_THREADS / nu : 0;
        const int iu0 = nu > 0 ? tid % nu : 0, iv0 = nu > 0 ? tid / nu : nv;
        for (int it = 0; it < a.ip.iters[l] && !stop; ++it) {
            __syncthreads();  // sH holds the current pose
            float R[9], t[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
#pragma unroll
                for (int k = 0; k < 3; ++k) R[3 * r + k] = (float)sH[4 * r + k];
                t[r] = (float)sH[4 * r + 3];
            }
            float acc[ICP_NS];
#pragma unroll
            for (int k = 0; k < ICP_NS; ++k) acc[k] = 0.f;
            int n_in = 0, n_valid = 0;
            float exit_hi[3], exit_lo[3];
            bool inside = true;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                exit_hi[k] = a.hi[k] - t[k];
                exit_lo[k] = t[k] - a.lo[k];
                inside = inside && exit_hi[k] > 0.f && exit_lo[k] > 0.f;
            }
            if (inside)  // the same for every thread of the block
                icp_sweep<true>(fr, a, iu0, iv0, du, dv, nu, nv, st, ifx, ify, R, t, exit_hi, exit_lo, dist2, acc,
                                n_in, n_valid);
            else
                icp_sweep<false>(fr, a, iu0, iv0, du, dv, nu, nv, st, ifx, ify, R, t, exit_hi, exit_lo, dist2, acc,
                                 n_in, n_valid);
            visited += (unsigned long long)n_valid;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int k = 0; k < ICP_NS; ++k) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], o);
                n_in += __shfl_down_sync(0xffffffffu, n_in, o);
                n_valid += __shfl_down_sync(0xffffffffu, n_valid, o);
            }
            if (lane == 0) {
#pragma unroll
                for (int k = 0; k < ICP_NS; ++k) s_part[w][k] = acc[k];
                s_cnt[w][0] = n_in;
                s_cnt[w][1] = n_valid;
            }
            __syncthreads();
            if (tid < ICP_NS) {
                double sum = 0.0;
                for (int ww = 0; ww < ICP_WARPS; ++ww) sum += (double)s_part[ww][tid];
                s_tot[tid] = sum;
            } else if (tid < ICP_NS + 2) {
                int sum = 0;
                for (int ww = 0; ww < ICP_WARPS; ++ww) sum += s_cnt[ww][tid - ICP_NS];
                s_n[tid - ICP_NS] = sum;
            }
            __syncthreads();
            if (tid == 0 && !icp_step(sH, s_tot, a.ip.ridge)) s_fail = 1;
            __syncthreads();
            stop = s_fail != 0;
        }
    }
    if (a.work && visited) atomicAdd(&a.work[W_ICP_PIX], visited);
    if (tid == 0) {
        const int nin = s_n[0], nval = s_n[1];
        const bool ok = !s_fail && nval > 0 && (double)nin >= a.ip.min_frac * (double)nval;
        const size_t o = (size_t)b * a.out_stride + c;
        a.ok[o] = ok ? 1 : 0;
        a.frac[o] = nval > 0 ? (float)((double)nin / (double)nval) : 0.f;
        if (ok)
            for (int q = 0; q < 12; ++q) P[q] = sH[q];
    }
}

// Where warps of different roles meet: __syncthreads() wants every thread of
// the block at one place of the program, a named barrier (1: __syncthreads()
// is 0) only THREADS of them at any.  Orders their memory accesses alike.
template <int THREADS>
__device__ __forceinline__ void role_barrier() {
    asm volatile("barrier.cta.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// The same by a cluster of C blocks per pose, for calls of few poses: the
// sums of the one-block kernel are serial chains of a thread (1,200 pixels at
// full resolution), so what they leave idle can only prepare their terms.
// Block c owns the chains of the one-block kernel's warps c OW, ... (OW = 8 /
// C streams, a lane per chain); its helper warps evaluate the streams'
// pixels ahead, a chunk at a time, and hand (depth, gap, direction, axis)
// over in shared memory, double-buffered with a barrier per chunk.  The
// owners add the terms in the same order and the lanes and warps are reduced
// in the same order, so the results do not depend on C.  Block 0 solves; the
// pose goes back through distributed shared memory.
//
// AX owner warps share a stream: one that branches on the face's axis, as the
// one-block kernel does, or one per axis, each with its nine sums and no
// branch.  Alone on an SM (C = 8) the owners are the critical path and three
// of them are faster (16 poses of 640x480: 423 us, 589 with one); with four
// blocks per SM (C = 4) instructions count and one that branches is (128
// poses: 877 us, 1010 without the branch).  About 150 us of either are the 11
// FP64 solves.  icp_blocks has when each pays.
template <int C, int AX>
struct IcpTeam {
    static constexpr int threads = C == 8 ? 32 * (AX + 9) : ICP_THREADS;
    static constexpr int loads = C == 8 ? 3 : ICP_LOADS;  // steps of a helper and chunk
};

template <int C, int AX>
__global__ void __cluster_dims__(C, 1, 1) __launch_bounds__(IcpTeam<C, AX>::threads, C == 8 ? 3 : 4)
    k_icp_team(IcpArgs a) {
    constexpr int OW = ICP_WARPS / C;             // streams of the block
    constexpr int NT = IcpTeam<C, AX>::threads;
    constexpr int HPS = (NT / 32 - OW * AX) / OW; // helper warps per stream
    constexpr int LD = IcpTeam<C, AX>::loads;
    constexpr int CH = HPS * LD;                  // steps of 32 pixels per stream and chunk
    __shared__ float4 s_a[2][OW][CH][32];         // depth, gap, direction x, y
    __shared__ float2 s_b[2][OW][CH][32];         // direction z, axis (-1: no inlier)
    __shared__ double sH[12];
    __shared__ float s_part[OW][ICP_NS];
    __shared__ int s_cnt[2];
    __shared__ double s_tot[ICP_NS];
    __shared__ int s_n[2];                        // inliers, valid pixels of the last iteration
    __shared__ int s_fail;
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int b = blockIdx.y, c = blockIdx.x / C;
    if (a.gate && a.gate[b] <= 0) return;         // the same for the whole cluster
    const int cnt = a.counts ? a.counts[b] : a.cap;
    if (c >= cnt) return;
    const Frame fr = a.frames[b];
    double *P = a.poses + ((size_t)b * a.pose_stride + c) * 12;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const bool owner = w < OW * AX;
    const int stream = w % OW, helper = (w - OW * AX) / OW, axis = w / OW;
    const int cell0 = (rank * OW + stream) * 32 + lane;  // the chain's first cell
    const int solver = 32 * ((c + b) & 3);        // spreads the poses' FP64 solves over the sub-partitions
    if (tid < 12) sH[tid] = P[tid];
    if (tid == 0) {
        s_fail = 0;
        s_n[0] = s_n[1] = 0;
        s_cnt[0] = s_cnt[1] = 0;
    }
    const float ifx = 1.0f / fr.fx, ify = 1.0f / fr.fy;
    unsigned long long visited = 0;
    bool stop = false;
    for (int l = 0; l < a.ip.levels && !stop; ++l) {
        const int st = a.ip.stride[l];
        const int nu = (fr.W + st - 1) / st, nv = (fr.H + st - 1) / st;
        const float dist2 = a.ip.dist[l] * a.ip.dist[l];
        const int steps = (nu * nv + ICP_THREADS - 1) / ICP_THREADS;
        const int chunks = (steps + CH - 1) / CH;
        // a helper's steps are HPS apart, its cells HPS * ICP_THREADS
        const int hop = HPS * ICP_THREADS;
        const int du = nu > 0 ? hop % nu : 0, dv = nu > 0 ? hop / nu : 0;
        const int hc = cell0 + (owner ? 0 : helper) * ICP_THREADS;
        const int iu0 = nu > 0 ? hc % nu : 0, iv0 = nu > 0 ? hc / nu : nv;
        for (int it = 0; it < a.ip.iters[l] && !stop; ++it) {
            __syncthreads();  // sH holds the current pose
            float R[9], t[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) {
#pragma unroll
                for (int k = 0; k < 3; ++k) R[3 * r + k] = (float)sH[4 * r + k];
                t[r] = (float)sH[4 * r + 3];
            }
            int n_in = 0, n_valid = 0;
            if (owner) {
                constexpr int NS = AX == 1 ? ICP_NS : 9;  // this warp's sums
                float acc[NS];
#pragma unroll
                for (int k = 0; k < NS; ++k) acc[k] = 0.f;
                // AXIS: the face axis of this warp's sums (all of them: -1)
                auto consume = [&](auto axis_t) {
                    constexpr int AXIS = decltype(axis_t)::value;
                    for (int ck = 0; ck <= chunks; ++ck) {
                        if (ck > 0) {
                            const int buf = (ck - 1) & 1;
#pragma unroll 4
                            for (int i = 0; i < CH; ++i) {
                                const float4 va = s_a[buf][stream][i][lane];
                                const float2 vb = s_b[buf][stream][i][lane];
                                const int ax = __float_as_int(vb.y);
                                if constexpr (AXIS < 0) {
                                    if (ax >= 0) icp_terms(ax, va.x, va.y, va.z, va.w, vb.x, acc);
                                } else {  // as icp_terms
                                    const float dir[3] = {va.z, va.w, vb.x};
                                    icp_add_axis(acc, ax == AXIS, __fmul_rn(va.x, dir[(AXIS + 2) % 3]),
                                                 -__fmul_rn(va.x, dir[(AXIS + 1) % 3]), __fmul_rn(va.y, dir[AXIS]));
                                }
                            }
                        }
                        role_barrier<NT>();
                    }
                };
                if constexpr (AX == 1)
                    consume(std::integral_constant<int, -1>());
                else if (axis == 0)
                    consume(std::integral_constant<int, 0>());
                else if (axis == 1)
                    consume(std::integral_constant<int, 1>());
                else
                    consume(std::integral_constant<int, 2>());
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int k = 0; k < NS; ++k) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], o);
                if (lane == 0)
#pragma unroll
                    for (int k = 0; k < NS; ++k) s_part[stream][(AX == 1 ? 0 : 9 * axis) + k] = acc[k];
            } else {
                float exit_hi[3], exit_lo[3];
                bool inside = true;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    exit_hi[k] = a.hi[k] - t[k];
                    exit_lo[k] = t[k] - a.lo[k];
                    inside = inside && exit_hi[k] > 0.f && exit_lo[k] > 0.f;
                }
                int iu = iu0, iv = iv0;
                for (int ck = 0; ck <= chunks; ++ck) {
                    if (ck < chunks) {
                        float dk[LD];
                        int uk[LD], vk[LD];
#pragma unroll
                        for (int j = 0; j < LD; ++j) {
                            uk[j] = iu * st;
                            vk[j] = iv * st;
                            dk[j] = iv < nv ? fr.depth[(size_t)vk[j] * fr.W + uk[j]] : 0.f;  // 0: no pixel
                            iu += du;
                            iv += dv;
                            if (iu >= nu) {
                                iu -= nu;
                                ++iv;
                            }
                        }
#pragma unroll
                        for (int j = 0; j < LD; ++j) {
                            float dir[3] = {0.f, 0.f, 0.f}, gap = 0.f;
                            const int ax = inside ? icp_gap<true>(a, dk[j], uk[j], vk[j], fr.cx, fr.cy, ifx, ify, R, t,
                                                                  exit_hi, exit_lo, dist2, dir, gap, n_valid)
                                                  : icp_gap<false>(a, dk[j], uk[j], vk[j], fr.cx, fr.cy, ifx, ify, R, t,
                                                                   exit_hi, exit_lo, dist2, dir, gap, n_valid);
                            n_in += ax >= 0;
                            const int i = j * HPS + helper;
                            s_a[ck & 1][stream][i][lane] = make_float4(dk[j], gap, dir[0], dir[1]);
                            s_b[ck & 1][stream][i][lane] = make_float2(dir[2], __int_as_float(ax));
                        }
                    }
                    role_barrier<NT>();
                }
                visited += (unsigned long long)n_valid;
                n_in = __reduce_add_sync(0xffffffffu, n_in);
                n_valid = __reduce_add_sync(0xffffffffu, n_valid);
                if (lane == 0) {
                    atomicAdd(&s_cnt[0], n_in);
                    atomicAdd(&s_cnt[1], n_valid);
                }
            }
            cluster.sync();  // every block's sums are there
            if (rank == 0) {
                if (tid < ICP_NS) {
                    double sum = 0.0;
                    for (int ww = 0; ww < ICP_WARPS; ++ww)
                        sum += (double)cluster.map_shared_rank(&s_part[0][0], ww / OW)[ww % OW * ICP_NS + tid];
                    s_tot[tid] = sum;
                } else if (tid < ICP_NS + 2) {
                    int sum = 0;
                    for (int r = 0; r < C; ++r) sum += cluster.map_shared_rank(s_cnt, r)[tid - ICP_NS];
                    s_n[tid - ICP_NS] = sum;
                }
                __syncthreads();
                if (tid == solver && !icp_step(sH, s_tot, a.ip.ridge)) s_fail = 1;
                __syncthreads();
                for (int e = tid; e < (C - 1) * 13; e += NT) {
                    const int r = e / 13 + 1, k = e % 13;
                    if (k < 12) cluster.map_shared_rank(sH, r)[k] = sH[k];
                    else *cluster.map_shared_rank(&s_fail, r) = s_fail;
                }
            }
            cluster.sync();  // the pose is back, the sums are read
            if (tid == 0) s_cnt[0] = s_cnt[1] = 0;
            stop = s_fail != 0;
        }
    }
    if (a.work && visited) atomicAdd(&a.work[W_ICP_PIX], visited);
    if (rank == 0 && tid == 0) {
        const int nin = s_n[0], nval = s_n[1];
        const bool ok = !s_fail && nval > 0 && (double)nin >= a.ip.min_frac * (double)nval;
        const size_t o = (size_t)b * a.out_stride + c;
        a.ok[o] = ok ? 1 : 0;
        a.frac[o] = nval > 0 ? (float)((double)nin / (double)nval) : 0.f;
        if (ok)
            for (int q = 0; q < 12; ++q) P[q] = sH[q];
    }
}

rl_status launch_icp(const IcpArgs &a, int n, cudaStream_t s) {
    if (n <= 0 || a.cap <= 0) return RL_OK;
    double cells = 0.0;  // pixels of an iteration, on average
    int iters = 0;
    for (int l = 0; l < a.ip.levels; ++l) {
        cells += (double)a.max_hw / (a.ip.stride[l] * a.ip.stride[l]) * a.ip.iters[l];
        iters += a.ip.iters[l];
    }
    switch (icp_blocks(a.resident, a.sm_count, (int64_t)a.cap * a.n_active, cells / iters)) {
    case 8: k_icp_team<8, 3><<<dim3(a.cap * 8, n), IcpTeam<8, 3>::threads, 0, s>>>(a); break;
    case 4: k_icp_team<4, 1><<<dim3(a.cap * 4, n), IcpTeam<4, 1>::threads, 0, s>>>(a); break;
    default: k_icp<<<dim3(a.cap, n), ICP_THREADS, 0, s>>>(a);
    }
    RL_LAUNCH_CK();
    return RL_OK;
}

template <int C, int AX>
static int resident_teams() {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(IcpTeam<C, AX>::threads);
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_icp_team<C, AX>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

const IcpResident &icp_resident(rl_scene *sc) {
    std::call_once(sc->icp_once, [sc] {
        sc->icp_resident.of8 = resident_teams<8, 3>();
        sc->icp_resident.of4 = resident_teams<4, 1>();
    });
    return sc->icp_resident;
}

}  // namespace rl
