// Really Quick Shift clustering of leaf reservoirs and the leaf mode store
// (Sec. 3.2.2, step 3); the leaf's reservoir is staged in shared memory.
// Compiled with --fmad=false.
//
// The clustering decisions (density order, parent within tau_c, nearest
// parent) are those of the FP64 definition: densities summed in index order
// from FP64 exp, squared distances in FP64.  GB300 issues an FP64 warp
// instruction every 64 cycles per sub-partition (1/64 of FP32), so the
// O(n^2) loops run in FP32 with a certified error bound and the FP64 value
// is taken only where the bound cannot decide:
//  - squared distances d2 in FP32 (fused): differences rounded once (u =
//    2^-24 relative), squares and sums 3 u more: within 5 u of the FP64
//    value.  Tests against tau_c^2 or against the nearest candidate so far
//    closer than 1e-6 relative are redone in FP64;
//  - densities: term t = 2^(d2 c), c = -log2(e) / (2 sigma^2) rounded, its
//    argument within 7 u relative, ex2.approx within 2^-22 relative; terms
//    summed in groups of 8 whose sums are Kahan-added, then over at most 32
//    lanes: within 14 u.  With x = -ln t the exact exponents,
//    |rho32 - rho64| <= 8 u sum(t x) + (14 u + 2^-22) rho, and sum(t x) <=
//    rho ln(n / rho) (the entropy bound, equality when all terms are equal);
//  - a comparison matters only between points within tau_c, and for point i
//    only if no point known to be denser is nearer; points at the same place
//    have the same density by definition.  The few points left get an FP64
//    density summed in any order (within 1e-13), and those still closer than
//    1e-12 relative one summed in index order, as the definition does.
// Cluster statistics and the covariance factor are FP64, members in index
// order, so the modes are identical to the FP64 definition's.
//
// Work split: one block per leaf.  S adjacent lanes share a point's row (S a
// power of two, as many as fit); with more rows than threads a thread takes
// two at a time, so that one shared-memory read serves two pairs.  The pairs
// within tau_c are collected as bit masks of 32 columns per lane first and
// compared afterwards: with a tenth of the columns near, nearly every warp
// would otherwise take the comparison branch on every column.  What bounds a
// full leaf (1024 points, about 0.2 ms on its SM): FP32 issue of the two pair
// loops (12 and 14 instructions a pair) and the FP64 sums of its clusters,
// which are serial by definition; those run one warp per cluster, 32 members'
// products computed by the lanes at once and the running sums on a lane each,
// so that a member costs two dependent FP64 additions instead of 27 FP64
// instructions of a warp.  A cluster of four blocks on each full leaf was
// slower (2.2 against 1.5 ms at that stage): the full leaves fill the GPU.
//
// Measured on GB300: 10,240 leaves of 107 points on average, about 1,200 of
// them full (24 frames of 640x480, 5 trees of depth 11, capacity 1024): 1.17
// ms, 13.7 ms with FP64 densities on single lanes and one thread per
// cluster's sums.  2,048 leaves of an online update, some 60 full: 0.29 ms,
// 5.4 ms before.
#include <type_traits>

#include "internal.h"

namespace rl {

struct RqsArgs {
    const float4 *res;
    const uint32_t *res_count;
    int kappa, m_max, min_cluster_size, n_leaves, fp16;
    double inv2s2, tau2, cov_eps;
    int64_t begin;
    uint8_t *nmodes;
    float4 *centroid;
    ushort4 *mpos_h;
    float4 *mpos_f;
    uchar4 *mrgb;
    float4 *mU;
    int32_t *msize;
};

// Upper Cholesky factor U (U^T U = S) of S = (cov + eps I)^-1.
__device__ void inverse_cov_factor(const double cv[6], double eps, double U[6]) {
    const double a = cv[0] + eps, b = cv[1], c = cv[2];
    const double d = cv[3] + eps, e = cv[4], f = cv[5] + eps;
    const double A = d * f - e * e, B = c * e - b * f, C = b * e - c * d;
    const double det = a * A + b * B + c * C;
    const double s00 = A / det, s01 = B / det, s02 = C / det;
    const double s11 = (a * f - c * c) / det, s12 = (b * c - a * e) / det;
    const double s22 = (a * d - b * b) / det;
    const double l00 = sqrt(s00);
    const double l10 = s01 / l00, l20 = s02 / l00;
    const double l11 = sqrt(s11 - l10 * l10);
    const double l21 = (s12 - l20 * l10) / l11;
    const double l22 = sqrt(s22 - l20 * l20 - l21 * l21);
    U[0] = l00; U[1] = l10; U[2] = l20; U[3] = l11; U[4] = l21; U[5] = l22;
}

__device__ __forceinline__ double dist2(const float4 a, const float4 b) {
    const double ex = (double)a.x - (double)b.x;
    const double ey = (double)a.y - (double)b.y;
    const double ez = (double)a.z - (double)b.z;
    return (ex * ex + ey * ey) + ez * ez;
}

__device__ __forceinline__ float dist2f(const float4 a, const float4 b) {
    const float ex = a.x - b.x, ey = a.y - b.y, ez = a.z - b.z;
    return fmaf(ez, ez, fmaf(ey, ey, ex * ex));
}

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

constexpr int RQS_THREADS = 512;
constexpr int RQS_STAT_WARPS = 8;       // warps of the FP64 sums (four sub-partitions, two each)
constexpr int RQS_BUF = 6 * 33;         // FP64 values per such warp: six rows of 32, odd stride

// Parzen rows of PP points p over the columns sub, sub + S, ...
template <int PP>
__device__ __forceinline__ void rqs_density(const float4 *pts, int n, float c2, const float4 (&p)[PP], int sub, int S,
                                            float (&rho)[PP]) {
    float comp[PP];
#pragma unroll
    for (int k = 0; k < PP; ++k) rho[k] = comp[k] = 0.f;
    auto add = [&](const float (&part)[PP]) {  // Kahan sum of the groups
#pragma unroll
        for (int k = 0; k < PP; ++k) {
            const float y = part[k] - comp[k];
            const float t = rho[k] + y;
            comp[k] = (t - rho[k]) - y;
            rho[k] = t;
        }
    };
    int j = sub;
    for (; j + 7 * S < n; j += 8 * S) {
        float part[PP];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float4 q = pts[j + u * S];
#pragma unroll
            for (int k = 0; k < PP; ++k) {
                const float t = ex2_approx(dist2f(p[k], q) * c2);
                part[k] = u == 0 ? t : part[k] + t;
            }
        }
        add(part);
    }
    if (j < n) {
        float part[PP];
#pragma unroll
        for (int k = 0; k < PP; ++k) part[k] = 0.f;
        for (; j < n; j += S) {
            const float4 q = pts[j];
#pragma unroll
            for (int k = 0; k < PP; ++k) part[k] += ex2_approx(dist2f(p[k], q) * c2);
        }
        add(part);
    }
}

// Shared state of the parent search.
struct RqsPar {
    const float4 *pts;
    const float *rho, *err;   // FP32 densities and their error bounds
    const double *rho64;      // FP64 densities of the points with need >= 1
    int *need;                // 1: FP64 density wanted, 2: summed in index order
    int *any;                 // set when a point's need is raised
    double tau2;
    float tau_lo, tau_hi;     // tau2 less / plus the FP32 margin
    int n;
};

// What a search does with a pair that the FP32 bounds cannot order.
enum RqsLevel {
    RQS_FP32,   // notes how near such a pair is
    RQS_MARK,   // raises the needs of those that are not farther than the parent found in FP32
    RQS_FP64,   // compares FP64 densities; closer than 1e-12: raises the needs to 2
    RQS_ORDER   // compares FP64 densities summed in index order
};

// b nearer to p than a (a < 0: no candidate yet); equal distances: lower index.
__device__ __forceinline__ bool rqs_nearer(const float4 *pts, const float4 p, int b, float db, int a, float da) {
    if (a < 0 || db < da * (1.f - 1e-6f)) return true;
    if (db > da * (1.f + 1e-6f)) return false;
    const double x = dist2(p, pts[b]), y = dist2(p, pts[a]);
    return x < y || (x == y && b < a);
}

// A point's search: its best parent so far, and the nearest undecided pair.
struct RqsBest {
    int j;
    float d2, und;
};

// Column j of point i, within tau_c up to the margin: a new nearest parent?
template <int LEVEL>
__device__ __forceinline__ void rqs_candidate(const RqsPar &r, const float4 p, int i, float ri, float ei, int j,
                                              RqsBest &o) {
    const float4 q = r.pts[j];
    const float d2 = dist2f(p, q);
    if (d2 >= r.tau_lo && dist2(p, q) > r.tau2) return;
    const float rj = r.rho[j];
    bool higher;
    if (fabsf(rj - ri) > (ei + r.err[j]) * 1.0001f) {
        higher = rj > ri;
    } else if (p.x == q.x && p.y == q.y && p.z == q.z && ri == ri) {  // one place, one density (a NaN has no order)
        higher = j < i;
    } else if (LEVEL == RQS_FP32) {
        o.und = fminf(o.und, d2);  // a NaN distance is never a parent's
        return;
    } else if (LEVEL == RQS_MARK) {
        if (o.j < 0 || !(d2 > o.d2 * (1.f + 1e-6f))) r.need[i] = r.need[j] = 1;
        return;
    } else {
        if (!r.need[j]) return;  // farther than a point known to be denser
        const double x = r.rho64[j], y = r.rho64[i];
        if (LEVEL == RQS_FP64 && !(fabs(x - y) > 1e-12 * y)) {
            r.need[i] = r.need[j] = 2;
            *r.any = 1;
            return;
        }
        higher = x > y || (x == y && j < i);
    }
    if (LEVEL != RQS_MARK && higher && rqs_nearer(r.pts, p, j, d2, o.j, o.d2)) {
        o.j = j;
        o.d2 = d2;
    }
}

// Parents of PP points (i[k] < 0: none) over the columns sub, sub + S, ...
template <int PP, int LEVEL>
__device__ __forceinline__ void rqs_parents(const RqsPar &r, const float4 (&p)[PP], const int (&i)[PP], int sub, int S,
                                            RqsBest (&o)[PP]) {
    float ri[PP], ei[PP];
#pragma unroll
    for (int k = 0; k < PP; ++k) {
        if (LEVEL != RQS_MARK) o[k] = {-1, 0.f, INFINITY};
        ri[k] = i[k] >= 0 ? r.rho[i[k]] : 0.f;
        ei[k] = i[k] >= 0 ? r.err[i[k]] : 0.f;
    }
    for (int j0 = sub; j0 < r.n; j0 += 32 * S) {
        uint32_t near[PP];
#pragma unroll
        for (int k = 0; k < PP; ++k) near[k] = 0;
        if (j0 + 31 * S < r.n) {
#pragma unroll
            for (int u = 0; u < 32; ++u) {
                const float4 q = r.pts[j0 + u * S];
#pragma unroll
                for (int k = 0; k < PP; ++k)
                    if (!(dist2f(p[k], q) > r.tau_hi)) near[k] |= 1u << u;
            }
        } else {
            for (int u = 0; j0 + u * S < r.n; ++u) {
                const float4 q = r.pts[j0 + u * S];
#pragma unroll
                for (int k = 0; k < PP; ++k)
                    if (!(dist2f(p[k], q) > r.tau_hi)) near[k] |= 1u << u;
            }
        }
#pragma unroll
        for (int k = 0; k < PP; ++k) {
            uint32_t m = i[k] >= 0 ? near[k] : 0u;
            while (m) {
                const int j = j0 + (__ffs(m) - 1) * S;
                m &= m - 1;
                if (j != i[k]) rqs_candidate<LEVEL>(r, p[k], i[k], ri[k], ei[k], j, o[k]);
            }
        }
    }
}

// Merges the candidates of the S lanes of a point.
__device__ __forceinline__ void rqs_merge(const float4 *pts, const float4 p, int S, RqsBest &o) {
    for (int off = 1; off < S; off <<= 1) {
        const int oj = __shfl_xor_sync(0xffffffffu, o.j, off);
        const float od = __shfl_xor_sync(0xffffffffu, o.d2, off);
        o.und = fminf(o.und, __shfl_xor_sync(0xffffffffu, o.und, off));
        if (oj >= 0 && rqs_nearer(pts, p, oj, od, o.j, o.d2)) {
            o.j = oj;
            o.d2 = od;
        }
    }
}

// Dynamic shared memory, per point: float4 pts, double rho64 (later the two
// int lists of the clusters), float rho and err, int parent, root, csize,
// need; then the FP64 buffers.
__global__ void __launch_bounds__(RQS_THREADS, 2) k_rqs(RqsArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int K = a.kappa + (a.kappa & 1);
    float4 *pts = (float4 *)smem;
    double *rho64 = (double *)(pts + K);
    float *rho = (float *)(rho64 + K);
    float *err = rho + K;
    int *parent = (int *)(err + K);
    int *root = parent + K;
    int *csize = root + K;
    int *need = csize + K;
    double *bufs = (double *)(need + K);  // [RQS_STAT_WARPS][RQS_BUF]
    // after the parents are known
    int *qual = (int *)rho64;             // [K] roots of the clusters large enough
    int *order = qual + K;                // [K] members of the kept clusters, by cluster
    __shared__ int n_qual, n_list, any;
    __shared__ int cl_root[64], cl_start[65];
    __shared__ double mu[64][3], cov[64][6];
    __shared__ float cen[3];

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int NT = RQS_THREADS;
    const int L = (int)((a.begin + blockIdx.x) % a.n_leaves);
    const uint32_t cnt = a.res_count[L];
    // fewer points than the smallest cluster: no modes
    const int n = cnt < (uint32_t)a.min_cluster_size ? 0 : (cnt < (uint32_t)a.kappa ? (int)cnt : a.kappa);

    for (int i = tid; i < n; i += NT) {
        pts[i] = a.res[(size_t)L * a.kappa + i];
        csize[i] = 0;
        need[i] = 0;
        rho64[i] = 0.0;
    }
    if (tid == 0) n_qual = n_list = any = 0;
    __syncthreads();
    int kept = 0;
    if (n > 0) {
        int S = 1;  // lanes per row
        while (S < 32 && 2 * S * n <= NT) S *= 2;
        const int slots = NT / S, sub = tid % S, slot = tid / S;
        const float c2 = (float)(-1.4426950408889634 * a.inv2s2);
        // rows i and i + slots: two at a time where the warp has both
        for (int i0 = slot; i0 - slot < n; i0 += 2 * slots) {
            const int wbase = i0 - (lane / S);  // the warp's first row
            if (wbase >= n) break;
            const int i1 = i0 + slots;
            float r[2];
            if (wbase + slots < n) {
                const float4 p[2] = {pts[min(i0, n - 1)], pts[min(i1, n - 1)]};
                rqs_density<2>(pts, n, c2, p, sub, S, r);
            } else {
                const float4 p[1] = {pts[min(i0, n - 1)]};
                float one[1];
                rqs_density<1>(pts, n, c2, p, sub, S, one);
                r[0] = one[0];
                r[1] = 0.f;
            }
            for (int off = 1; off < S; off <<= 1) {
                r[0] += __shfl_xor_sync(0xffffffffu, r[0], off);
                r[1] += __shfl_xor_sync(0xffffffffu, r[1], off);
            }
            if (sub == 0) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int i = k ? i1 : i0;
                    if (i >= n) continue;
                    // the bound of the file comment (4.8e-7 and 1.08e-6)
                    // with 2% for its own rounding and second-order terms
                    const float ln = fmaxf(logf((float)n / r[k]), 0.f) + 0.01f;
                    const float e = r[k] * (4.9e-7f * ln + 1.1e-6f) + 1e-30f * (float)n;
                    rho[i] = r[k];
                    err[i] = e;
                }
            }
        }
        __syncthreads();
        // Parent: nearest point of higher density within tau_c (ties:
        // lower index).  Rows whose nearest undecided pair is not farther
        // than the parent found in FP32 are listed in `root`.
        const float tau2f = (float)a.tau2;
        const RqsPar rp{pts, rho, err, rho64, need, &any, a.tau2, tau2f * (1.f - 1.2e-6f), tau2f * (1.f + 1.2e-6f),
                        n};
        auto found = [&](int i, const RqsBest &o) {
            parent[i] = o.j;
            if (o.und < INFINITY && (o.j < 0 || !(o.und > o.d2 * (1.f + 1e-6f)))) root[atomicAdd(&n_list, 1)] = i;
        };
        for (int i0 = slot; i0 - slot < n; i0 += 2 * slots) {
            const int wbase = i0 - (lane / S);
            if (wbase >= n) break;
            const int i1 = i0 + slots;
            if (wbase + slots < n) {
                const float4 p[2] = {pts[min(i0, n - 1)], pts[min(i1, n - 1)]};
                const int id[2] = {i0 < n ? i0 : -1, i1 < n ? i1 : -1};
                RqsBest o[2];
                rqs_parents<2, RQS_FP32>(rp, p, id, sub, S, o);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    rqs_merge(pts, p[k], S, o[k]);
                    if (sub == 0 && id[k] >= 0) found(id[k], o[k]);
                }
            } else {
                const float4 p[1] = {pts[min(i0, n - 1)]};
                const int id[1] = {i0 < n ? i0 : -1};
                RqsBest o[1];
                rqs_parents<1, RQS_FP32>(rp, p, id, sub, S, o);
                rqs_merge(pts, p[0], S, o[0]);
                if (sub == 0 && id[0] >= 0) found(id[0], o[0]);
            }
        }
        __syncthreads();
        const int listed = n_list;
        if (listed > 0) {
            // a warp per listed row: marks the points to be known in FP64
            for (int e = w; e < listed; e += NT / 32) {
                const int id[1] = {root[e]};
                const float4 p[1] = {pts[id[0]]};
                RqsBest o[1] = {{parent[id[0]], 0.f, 0.f}};
                if (o[0].j >= 0) o[0].d2 = dist2f(p[0], pts[o[0].j]);
                rqs_parents<1, RQS_MARK>(rp, p, id, lane, 32, o);
            }
            __syncthreads();
            // their FP64 densities, by all threads, summed in any order
            for (int b0 = 0; b0 < n; b0 += 32)
                for (unsigned m = __ballot_sync(0xffffffffu, b0 + lane < n && need[b0 + lane]); m; m &= m - 1) {
                    const int i = b0 + __ffs(m) - 1;
                    const float4 p = pts[i];
                    double r = 0.0;
                    for (int j = tid; j < n; j += NT) r += exp(-(dist2(p, pts[j]) * a.inv2s2));
#pragma unroll
                    for (int off = 16; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
                    if (lane == 0) atomicAdd(&rho64[i], r);
                }
            __syncthreads();
            auto again = [&](auto level) {
                for (int e = w; e < listed; e += NT / 32) {
                    const int id[1] = {root[e]};
                    const float4 p[1] = {pts[id[0]]};
                    RqsBest o[1];
                    rqs_parents<1, decltype(level)::value>(rp, p, id, lane, 32, o);
                    rqs_merge(pts, p[0], 32, o[0]);
                    if (lane == 0) parent[id[0]] = o[0].j;
                }
            };
            again(std::integral_constant<int, RQS_FP64>());
            __syncthreads();
            if (any) {  // densities within 1e-12: summed as the definition sums them
                if (w < RQS_STAT_WARPS)
                    for (int i0 = w; i0 < n; i0 += RQS_STAT_WARPS) {
                        if (need[i0] != 2) continue;
                        double *buf = bufs + w * RQS_BUF;
                        const float4 p = pts[i0];
                        double r = 0.0;
                        for (int j0 = 0; j0 < n; j0 += 32) {
                            if (j0 + lane < n) buf[lane] = exp(-(dist2(p, pts[j0 + lane]) * a.inv2s2));
                            __syncwarp();
                            const int m = min(32, n - j0);
                            for (int k = 0; k < m; ++k) r += buf[k];
                            __syncwarp();
                        }
                        if (lane == 0) rho64[i0] = r;
                    }
                __syncthreads();
                again(std::integral_constant<int, RQS_ORDER>());
            }
        }
        __syncthreads();
        for (int i = tid; i < n; i += NT) {
            int r = i;
            while (parent[r] >= 0) r = parent[r];
            root[i] = r;
            atomicAdd(&csize[r], 1);
        }
        __syncthreads();
        // Rank the qualifying clusters by (size desc, root asc).
        for (int r = tid; r < n; r += NT)
            if (parent[r] < 0 && csize[r] >= a.min_cluster_size) qual[atomicAdd(&n_qual, 1)] = r;
        __syncthreads();
        const int nq = n_qual;
        for (int e = tid; e < nq; e += NT) {
            const int r = qual[e], sr = csize[r];
            int rk = 0;
            for (int f = 0; f < nq; ++f) {
                const int o = qual[f], so = csize[o];
                rk += so > sr || (so == sr && o < r);
            }
            if (rk < a.m_max) cl_root[rk] = r;
        }
        __syncthreads();
        kept = min(nq, a.m_max);
        if (w == 0) {  // first member of each kept cluster in `order`
            int s0 = lane < kept ? csize[cl_root[lane]] : 0, s1 = lane + 32 < kept ? csize[cl_root[lane + 32]] : 0;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int t0 = __shfl_up_sync(0xffffffffu, s0, off), t1 = __shfl_up_sync(0xffffffffu, s1, off);
                if (lane >= off) {
                    s0 += t0;
                    s1 += t1;
                }
            }
            s1 += __shfl_sync(0xffffffffu, s0, 31);
            cl_start[lane + 1] = s0;
            cl_start[lane + 33] = s1;
            if (lane == 0) cl_start[0] = 0;
        }
        __syncthreads();
        // Per-cluster statistics, members summed in index order, a warp each.
        if (w < RQS_STAT_WARPS)
            for (int k = w; k < kept; k += RQS_STAT_WARPS) {
                double *buf = bufs + w * RQS_BUF;
                const int r = cl_root[k], c = cl_start[k + 1] - cl_start[k];
                int *mem = order + cl_start[k];
                for (int i0 = 0, f = 0; f < c; i0 += 32) {
                    const unsigned in = __ballot_sync(0xffffffffu, i0 + lane < n && root[i0 + lane] == r);
                    if (in >> lane & 1u) mem[f + __popc(in & ((1u << lane) - 1u))] = i0 + lane;
                    f += __popc(in);
                }
                __syncwarp();
                double s = 0.0;  // lane q: the q-th running sum
                unsigned sr = 0, sg = 0, sb = 0;
                for (int f = 0; f < c; f += 32) {
                    const int m = min(32, c - f);
                    if (lane < m) {
                        const float4 p = pts[mem[f + lane]];
                        buf[lane] = (double)p.x;
                        buf[33 + lane] = (double)p.y;
                        buf[66 + lane] = (double)p.z;
                        const uint32_t rgb = __float_as_uint(p.w);
                        sr += rgb & 255;
                        sg += (rgb >> 8) & 255;
                        sb += (rgb >> 16) & 255;
                    }
                    __syncwarp();
                    if (lane < 3)
                        for (int e = 0; e < m; ++e) s += buf[33 * lane + e];
                    __syncwarp();
                }
                const double mean = s / c;
                const double m0 = __shfl_sync(0xffffffffu, mean, 0), m1 = __shfl_sync(0xffffffffu, mean, 1),
                             m2 = __shfl_sync(0xffffffffu, mean, 2);
                s = 0.0;
                for (int f = 0; f < c; f += 32) {
                    const int m = min(32, c - f);
                    if (lane < m) {
                        const float4 p = pts[mem[f + lane]];
                        const double e0 = (double)p.x - m0, e1 = (double)p.y - m1, e2 = (double)p.z - m2;
                        buf[lane] = e0 * e0;
                        buf[33 + lane] = e0 * e1;
                        buf[66 + lane] = e0 * e2;
                        buf[99 + lane] = e1 * e1;
                        buf[132 + lane] = e1 * e2;
                        buf[165 + lane] = e2 * e2;
                    }
                    __syncwarp();
                    if (lane < 6)
                        for (int e = 0; e < m; ++e) s += buf[33 * lane + e];
                    __syncwarp();
                }
                if (lane < 6) cov[k][lane] = c > 1 ? s / (double)(c - 1) : 0.0;
                if (lane < 3) mu[k][lane] = mean;
                sr = __reduce_add_sync(0xffffffffu, sr);
                sg = __reduce_add_sync(0xffffffffu, sg);
                sb = __reduce_add_sync(0xffffffffu, sb);
                if (lane == 0) {
                    const size_t e = (size_t)L * a.m_max + k;
                    const unsigned h = (unsigned)c / 2, d = (unsigned)c;
                    a.mrgb[e] = make_uchar4((uint8_t)((sr + h) / d), (uint8_t)((sg + h) / d),
                                            (uint8_t)((sb + h) / d), 0);
                    a.msize[e] = c;
                }
            }
        __syncthreads();
        if (tid < kept) {
            double U[6];
            inverse_cov_factor(cov[tid], a.cov_eps, U);
            const size_t e = (size_t)L * a.m_max + tid;
            a.mU[2 * e] = make_float4((float)U[0], (float)U[1], (float)U[2], (float)U[3]);
            a.mU[2 * e + 1] = make_float4((float)U[4], (float)U[5], 0.f, 0.f);
        }
    }
    // Per-leaf FP32 centroid of the kept modes; positions as FP16 offsets.
    if (w == NT / 32 - 1 && lane < 3) {
        double c = 0;
        for (int k = 0; k < kept; ++k) c += mu[k][lane];
        cen[lane] = kept > 0 ? (float)(c / kept) : 0.f;
    }
    __syncthreads();
    if (tid == 0) {
        a.centroid[L] = make_float4(cen[0], cen[1], cen[2], 0.f);
        a.nmodes[L] = (uint8_t)kept;
    }
    for (int k = tid; k < a.m_max; k += NT) {
        const size_t e = (size_t)L * a.m_max + k;
        if (k >= kept) {
            if (a.fp16) a.mpos_h[e] = make_ushort4(0, 0, 0, 0);
            else a.mpos_f[e] = make_float4(0, 0, 0, 0);
            a.mrgb[e] = make_uchar4(0, 0, 0, 0);
            a.mU[2 * e] = make_float4(0, 0, 0, 0);
            a.mU[2 * e + 1] = make_float4(0, 0, 0, 0);
            a.msize[e] = 0;
            continue;
        }
        if (a.fp16) {
            const __half hx = __double2half(mu[k][0] - (double)cen[0]);
            const __half hy = __double2half(mu[k][1] - (double)cen[1]);
            const __half hz = __double2half(mu[k][2] - (double)cen[2]);
            a.mpos_h[e] = make_ushort4(__half_as_ushort(hx), __half_as_ushort(hy),
                                       __half_as_ushort(hz), 0);
        } else {
            a.mpos_f[e] = make_float4((float)mu[k][0], (float)mu[k][1], (float)mu[k][2], 0.f);
        }
    }
}

static size_t rqs_smem(int kappa) {
    const size_t K = (size_t)kappa + (kappa & 1);
    return K * (sizeof(float4) + sizeof(double) + 2 * sizeof(float) + 4 * sizeof(int)) +
           RQS_STAT_WARPS * RQS_BUF * sizeof(double);
}

rl_status update_modes(rl_forest *f, int64_t begin, int64_t count, cudaStream_t s) {
    if (count <= 0) return RL_OK;
    const rl_forest_params &p = f->p;
    RqsArgs a;
    a.res = f->res;
    a.res_count = f->res_count;
    a.kappa = p.kappa;
    a.m_max = p.m_max;
    a.min_cluster_size = p.min_cluster_size;
    a.n_leaves = f->n_leaves;
    a.fp16 = p.mode_precision == RL_MODES_FP16_OFFSET;
    const double sg = (double)p.sigma, tc = (double)p.tau_c;
    a.inv2s2 = 1.0 / (2.0 * sg * sg);
    a.tau2 = tc * tc;
    a.cov_eps = (double)p.cov_eps;
    a.begin = begin;
    a.nmodes = f->nmodes;
    a.centroid = f->centroid;
    a.mpos_h = f->mpos_h;
    a.mpos_f = f->mpos_f;
    a.mrgb = f->mrgb;
    a.mU = f->mU;
    a.msize = f->msize;
    const size_t sm = rqs_smem(p.kappa);
    RL_CK(cudaFuncSetAttribute(k_rqs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    // Grid dimension x is limited to 2^31-1; leaves per launch are chunked.
    for (int64_t off = 0; off < count; off += (1 << 30)) {
        const int64_t n = count - off < (1 << 30) ? count - off : (1 << 30);
        a.begin = begin + off;
        k_rqs<<<(unsigned)n, RQS_THREADS, sm, s>>>(a);
        RL_LAUNCH_CK();
    }
    return RL_OK;
}

}  // namespace rl
