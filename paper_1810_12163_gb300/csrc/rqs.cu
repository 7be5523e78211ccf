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
//    summed in groups of 8 whose sums are Kahan-added: within 14 u.  With x = -ln t the exact exponents,
//    |rho32 - rho64| <= 8 u sum(t x) + (14 u + 2^-22) rho, and sum(t x) <=
//    rho ln(n / rho) (the entropy bound, equality when all terms are equal).
//    Terms below 2^-40 are left out where whole tiles of points are that far
//    apart; they add at most n 2^-40;
//  - a comparison matters only between points within tau_c, and for point i
//    only if no point known to be denser is nearer; points at the same place
//    have the same density by definition.  The few points left get an FP64
//    density summed in any order (within 1e-13), and those still closer than
//    1e-12 relative one summed in index order, as the definition does.
// Cluster statistics and the covariance factor are FP64, members in index
// order, so the modes are identical to the FP64 definition's.
//
// Work split: one block per leaf.  The points are sorted along a Morton curve;
// a warp takes 32 of them as rows, a lane each, and the groups of 8 columns
// whose boxes are near enough to matter (0.74 m at sigma = 0.1 m for the
// densities, tau_c for the parents): in a full leaf most are not.  A row's
// own groups come first, so that its parent is soon found and columns farther
// off or surely less dense are passed over by two comparisons; the others are
// noted as a bit mask first and compared afterwards, since with one column in
// ten near nearly every warp would otherwise take the comparison branch on
// every column.  The clusters' FP64 sums run eight lanes a cluster, the four
// clusters of a warp sharing its FP64 instructions.  The means are exact sums
// wherever the values' bits span at most 53, and then any order will do;
// otherwise, and for the covariances, the sums are serial by definition: the
// lanes compute eight members' products at once, then carry a running sum
// each (a warp per cluster took three FP64 instructions a member, a thread
// per cluster 27).
// Thousands of cycles of a leaf of more than 600 points, training / online
// (where clusters are larger), by clock stamps at the phases' barriers: sort
// and boxes 22 / 19, densities 50 / 62, parents 62 / 71, FP64 densities 16 /
// 10, FP64 comparisons 15 / 7, members 9 / 15, cluster sums 26 / 58, factors
// 11 / 10.  With the columns in groups of 32, every column of a group compared
// and a warp per cluster it was 297 and 350 in all.  A cluster of four blocks
// on each full leaf was slower in training, where the full leaves fill the
// GPU; online, where they do not, it was not tried.
//
// Measured on GB300: 10,240 leaves of 107 points on average, about 800 of
// more than 600 (24 frames of 640x480, 5 trees of depth 11, capacity 1024):
// 0.67 ms; 1.17 ms with every pair of points looked at, 13.7 ms with FP64
// densities on single lanes and one thread per cluster's sums.  2,048 leaves
// of an online update, some 35 of more than 600 points: 0.20 ms, 0.29 ms and
// 5.4 ms before; the largest leaf's serial parts bound that.  1,024 threads a
// block: 1.05 and 0.20 ms.
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
constexpr int RQS_GROUP = 8;            // columns with a box of their own

// Squared distance between two boxes (0 if they meet), a little
// below the exact value.
__device__ __forceinline__ float box_gap2(const float4 alo, const float4 ahi, const float4 blo, const float4 bhi) {
    const float x = fmaxf(0.f, fmaxf(blo.x - ahi.x, alo.x - bhi.x));
    const float y = fmaxf(0.f, fmaxf(blo.y - ahi.y, alo.y - bhi.y));
    const float z = fmaxf(0.f, fmaxf(blo.z - ahi.z, alo.z - bhi.z));
    return fmaf(z, z, fmaf(y, y, x * x)) * 0.9999f;
}

// Morton code of 7 + 7 + 6 bits.
__device__ __forceinline__ uint32_t morton20(uint32_t x, uint32_t y, uint32_t z) {
    uint32_t m = 0;
#pragma unroll
    for (int b = 0; b < 7; ++b) {
        m |= (x >> b & 1u) << (3 * b + 1);
        m |= (y >> b & 1u) << (3 * b);
        if (b < 6) m |= (z >> b & 1u) << (3 * b + 2);
    }
    return m;
}

// Calls f(g) for the column groups of row tile `mine`, then for every other
// group whose box is within `cut` (squared) of the tile's; every lane of the
// warp together.
template <class F>
__device__ __forceinline__ void near_groups(const float4 *box, int groups, int mine, float cut, F f) {
    constexpr int PER = 32 / RQS_GROUP;
    const int lane = threadIdx.x & 31, g0 = PER * mine, g1 = min(g0 + PER, groups);
    float4 lo = box[2 * g0], hi = box[2 * g0 + 1];
    for (int g = g0 + 1; g < g1; ++g) {
        const float4 l = box[2 * g], h = box[2 * g + 1];
        lo = make_float4(fminf(lo.x, l.x), fminf(lo.y, l.y), fminf(lo.z, l.z), 0.f);
        hi = make_float4(fmaxf(hi.x, h.x), fmaxf(hi.y, h.y), fmaxf(hi.z, h.z), 0.f);
    }
    for (int t0 = -32; t0 < groups; t0 += 32) {
        unsigned m;
        if (t0 < 0) {
            m = (1u << (g1 - g0)) - 1u;
        } else {
            const int g = t0 + lane, gc = min(g, groups - 1);
            m = __ballot_sync(0xffffffffu, g < groups && (g < g0 || g >= g1) &&
                                               !(box_gap2(lo, hi, box[2 * gc], box[2 * gc + 1]) > cut));
        }
        for (const int base = t0 < 0 ? g0 : t0; m; m &= m - 1) f(base + __ffs(m) - 1);
    }
}

// (double)x by its bits: conversions take the FP64 pipe.
__device__ __forceinline__ double widen(float x) {
    const uint32_t b = __float_as_uint(x);
    if ((b >> 23 & 255u) - 1u < 254u)
        return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
    return (double)x;  // zero, subnormal, not finite
}

// Exponents of the values other than zero of a sum.
struct Span {
    int lo = 255, hi = 0;
    __device__ void add(float x) {
        const uint32_t b = __float_as_uint(x) & 0x7fffffffu;
        const int e = max((int)(b >> 23), 1);
        if (b) {
            lo = min(lo, e);
            hi = max(hi, e);
        }
    }
    __device__ void join(int o) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    // all partial sums of n of them are multiples of 2^(lo - 150) below n 2^(hi - 126)
    __device__ bool exact(int n) const { return hi - lo + (32 - __clz(n)) <= 29; }
};

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

// A point's search by a warp, lane by lane of the columns in index order.
template <int LEVEL>
__device__ __forceinline__ void rqs_row(const RqsPar &r, int i, RqsBest &o) {
    const int lane = threadIdx.x & 31;
    const float4 p = r.pts[i];
    const float ri = r.rho[i], ei = r.err[i];
    if (LEVEL != RQS_MARK) o = {-1, 0.f, INFINITY};
    for (int j = lane; j < r.n; j += 32)
        if (j != i && !(dist2f(p, r.pts[j]) > r.tau_hi)) rqs_candidate<LEVEL>(r, p, i, ri, ei, j, o);
    if constexpr (LEVEL != RQS_MARK) {
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int oj = __shfl_xor_sync(0xffffffffu, o.j, off);
            const float od = __shfl_xor_sync(0xffffffffu, o.d2, off);
            if (oj >= 0 && rqs_nearer(r.pts, p, oj, od, o.j, o.d2)) {
                o.j = oj;
                o.d2 = od;
            }
        }
    }
}

// Dynamic shared memory, per point: float4 pts, 16 bytes that hold the sorted
// copy spts (x, y, z, an upper bound of the density) and later double rho64
// (then the two int lists of the clusters), int root and csize; float rho and
// err (first the sort keys), int parent and need; two float4 box per group of
// columns; then the FP64 buffers.
__global__ void __launch_bounds__(RQS_THREADS, 2) k_rqs(RqsArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int K = (a.kappa + 31) & ~31;
    float4 *pts = (float4 *)smem;
    float4 *spts = pts + K;
    double *rho64 = (double *)spts;
    int *root = (int *)(rho64 + K);
    int *csize = root + K;
    float *rho = (float *)(spts + K);
    float *err = rho + K;
    uint32_t *keys = (uint32_t *)rho;     // [2 K]
    int *parent = (int *)(err + K);
    int *need = parent + K;
    float4 *box = (float4 *)(need + K);   // [K / RQS_GROUP][2]
    double *bufs = (double *)(box + K / RQS_GROUP * 2);  // [RQS_STAT_WARPS][RQS_BUF]
    // until the parents are known: index of the sorted point k in the low half of need[k]
    uint16_t *sorted = (uint16_t *)need;
    uint8_t *open = (uint8_t *)need;      // [4 i + 3]: point i's parent is not decided
    // after the parents are known
    int *qual = (int *)rho64;             // [K] roots of the clusters large enough
    int *order = qual + K;                // [K] members of the kept clusters, by cluster
    __shared__ int n_qual, n_list, n_near, any;
    __shared__ int cl_root[64], cl_start[65];
    __shared__ double mu[64][3], cov[64][6];
    __shared__ float cen[3];

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int NT = RQS_THREADS;
    const int L = (int)((a.begin + blockIdx.x) % a.n_leaves);
    const uint32_t cnt = a.res_count[L];
    // fewer points than the smallest cluster: no modes
    const int n = cnt < (uint32_t)a.min_cluster_size ? 0 : (cnt < (uint32_t)a.kappa ? (int)cnt : a.kappa);

    float3 mn = make_float3(INFINITY, INFINITY, INFINITY), mx = make_float3(-INFINITY, -INFINITY, -INFINITY);
    bool finite = true;
    for (int i = tid; i < n; i += NT) {
        const float4 p = a.res[(size_t)L * a.kappa + i];
        pts[i] = p;
        mn = make_float3(fminf(mn.x, p.x), fminf(mn.y, p.y), fminf(mn.z, p.z));
        mx = make_float3(fmaxf(mx.x, p.x), fmaxf(mx.y, p.y), fmaxf(mx.z, p.z));
        finite = finite && isfinite(p.x) && isfinite(p.y) && isfinite(p.z);
    }
    if (tid == 0) n_qual = n_list = n_near = any = 0;
    int kept = 0;
    if (n > 0) {
        // ---- tiles of 32 points along a Morton curve (few points: as they are)
        const int n_tiles = (n + 31) / 32, n32 = n_tiles * 32;
        int P2 = 64;
        while (P2 < n) P2 *= 2;
        if (n > 64) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                mn = make_float3(fminf(mn.x, __shfl_xor_sync(0xffffffffu, mn.x, o)),
                                 fminf(mn.y, __shfl_xor_sync(0xffffffffu, mn.y, o)),
                                 fminf(mn.z, __shfl_xor_sync(0xffffffffu, mn.z, o)));
                mx = make_float3(fmaxf(mx.x, __shfl_xor_sync(0xffffffffu, mx.x, o)),
                                 fmaxf(mx.y, __shfl_xor_sync(0xffffffffu, mx.y, o)),
                                 fmaxf(mx.z, __shfl_xor_sync(0xffffffffu, mx.z, o)));
            }
            float4 *ext = (float4 *)bufs;  // of the warps
            if (lane == 0) {
                ext[2 * w] = make_float4(mn.x, mn.y, mn.z, 0.f);
                ext[2 * w + 1] = make_float4(mx.x, mx.y, mx.z, 0.f);
            }
            __syncthreads();
            for (int k = 0; k < NT / 32; ++k) {
                const float4 l = ext[2 * k], h = ext[2 * k + 1];
                mn = make_float3(fminf(mn.x, l.x), fminf(mn.y, l.y), fminf(mn.z, l.z));
                mx = make_float3(fmaxf(mx.x, h.x), fmaxf(mx.y, h.y), fmaxf(mx.z, h.z));
            }
            const float sx = 127.99f / fmaxf(mx.x - mn.x, 1e-6f), sy = 127.99f / fmaxf(mx.y - mn.y, 1e-6f),
                        sz = 63.99f / fmaxf(mx.z - mn.z, 1e-6f);
            for (int i = tid; i < P2; i += NT) {
                uint32_t key = 0xFFFFFFFFu;
                if (i < n) {
                    const float4 p = pts[i];
                    const uint32_t x = (uint32_t)min(max((int)((p.x - mn.x) * sx), 0), 127),
                                   y = (uint32_t)min(max((int)((p.y - mn.y) * sy), 0), 127),
                                   z = (uint32_t)min(max((int)((p.z - mn.z) * sz), 0), 63);
                    key = morton20(x, y, z) << 12 | (uint32_t)i;
                }
                keys[i] = key;
            }
            __syncthreads();
            // bitonic sort, strides below 32 within a warp
            auto in_warp = [&](int k0, int k1) {
                for (int i = tid; i < P2; i += NT) {
                    uint32_t x = keys[i];
                    for (int k = k0; k <= k1; k <<= 1)
                        for (int j = min(k >> 1, 16); j > 0; j >>= 1) {
                            const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
                            x = ((i & k) == 0) == ((i & j) == 0) ? min(x, y) : max(x, y);
                        }
                    keys[i] = x;
                }
                __syncthreads();
            };
            in_warp(2, 32);
            for (int k = 64; k <= P2; k <<= 1) {
                for (int j = k >> 1; j >= 32; j >>= 1) {
                    for (int e = tid; e < P2 / 2; e += NT) {
                        const int i = 2 * e - (e & (j - 1));
                        const uint32_t x = keys[i], y = keys[i + j];
                        if ((x > y) == ((i & k) == 0)) {
                            keys[i] = y;
                            keys[i + j] = x;
                        }
                    }
                    __syncthreads();
                }
                in_warp(k, k);
            }
        } else {
            __syncthreads();
        }
        for (int k = tid; k < n32; k += NT) {
            const int i = k < n ? (n > 64 ? (int)(keys[k] & 4095u) : k) : -1;
            // padding: so far off that its terms are 0
            const float4 p = i >= 0 ? pts[i] : make_float4(3e38f, 3e38f, 3e38f, 0.f);
            spts[k] = make_float4(p.x, p.y, p.z, 0.f);
            need[k] = i & 0xFFFF;
        }
        // every group counts where a point is not finite (its distances have no order)
        const bool all = !__syncthreads_and(finite);
        const int groups = (n + RQS_GROUP - 1) / RQS_GROUP;
        for (int t = w; t < n_tiles; t += NT / 32) {
            const float4 p = spts[min(t * 32 + lane, n - 1)];
            float4 lo = p, hi = p;
#pragma unroll
            for (int o = 1; o < RQS_GROUP; o <<= 1) {
                lo = make_float4(fminf(lo.x, __shfl_xor_sync(0xffffffffu, lo.x, o)),
                                 fminf(lo.y, __shfl_xor_sync(0xffffffffu, lo.y, o)),
                                 fminf(lo.z, __shfl_xor_sync(0xffffffffu, lo.z, o)), 0.f);
                hi = make_float4(fmaxf(hi.x, __shfl_xor_sync(0xffffffffu, hi.x, o)),
                                 fmaxf(hi.y, __shfl_xor_sync(0xffffffffu, hi.y, o)),
                                 fmaxf(hi.z, __shfl_xor_sync(0xffffffffu, hi.z, o)), 0.f);
            }
            const int g = (t * 32 + lane) / RQS_GROUP;
            if (lane % RQS_GROUP == 0 && g < groups) {
                box[2 * g] = lo;
                box[2 * g + 1] = hi;
            }
        }
        __syncthreads();
        // ---- densities (the sort keys are no longer needed)
        const float c2 = fminf((float)(-1.4426950408889634 * a.inv2s2), -1.2e-38f);
        const float cut = all ? INFINITY : -40.f / c2 * 1.0001f;  // terms beyond are below 2^-40
        for (int t = w; t < n_tiles; t += NT / 32) {
            const int k = t * 32 + lane;
            const float4 p = spts[k];
            float sum = 0.f, comp = 0.f;
            near_groups(box, groups, t, cut, [&](int g) {
                float part = 0.f;
#pragma unroll
                for (int u = 0; u < RQS_GROUP; ++u) {
                    const float e = ex2_approx(dist2f(p, spts[g * RQS_GROUP + u]) * c2);
                    part = u == 0 ? e : part + e;
                }
                const float yk = part - comp;  // Kahan sum of the groups
                const float tk = sum + yk;
                comp = (tk - sum) - yk;
                sum = tk;
            });
            if (k < n) {
                const int i = sorted[2 * k];
                // the bound of the file comment (8 u = 4.77e-7, 14 u + 2^-22 =
                // 1.07e-6) with 2% for its own rounding and second-order terms
                const float ln = fmaxf(logf((float)n / sum), 0.f) + 0.01f;
                const float e = sum * (4.9e-7f * ln + 1.1e-6f) + 1e-12f * (float)n;
                rho[i] = sum;
                err[i] = e;
                spts[k].w = sum + 1.2f * e;  // exceeds rho + err by more than its rounding
            }
        }
        __syncthreads();
        // ---- parent: nearest point of higher density within tau_c (ties:
        // lower index).  A row whose nearest undecided pair is not farther
        // than the parent found in FP32 is noted in `need`.
        const float tau2f = (float)a.tau2;
        const RqsPar rp{pts, rho, err, rho64, need, &any, a.tau2, tau2f * (1.f - 1.2e-6f), tau2f * (1.f + 1.2e-6f),
                        n};
        const float tcut = all ? INFINITY : rp.tau_hi;
        for (int t = w; t < n_tiles; t += NT / 32) {
            const int k = t * 32 + lane, i = k < n ? sorted[2 * k] : 0;
            const float4 p = spts[k];
            const float ri = rho[i], ei = err[i], least = ri - 1.2f * ei;
            RqsBest o = {-1, 0.f, INFINITY};
            float most = k < n ? rp.tau_hi : -1.f;  // candidates beyond are not nearer than the best so far
            near_groups(box, groups, t, tcut, [&](int g) {
                uint32_t near = 0;
#pragma unroll
                for (int u = 0; u < RQS_GROUP; ++u) {
                    const float4 q = spts[g * RQS_GROUP + u];
                    if (!(dist2f(p, q) > most) && !(q.w < least)) near |= 1u << u;  // a NaN goes on
                }
                if (k >= n) near = 0;
                for (; near; near &= near - 1) {
                    const int c = g * RQS_GROUP + __ffs(near) - 1;
                    if (c == k || c >= n) continue;
                    rqs_candidate<RQS_FP32>(rp, p, i, ri, ei, sorted[2 * c], o);
                    if (o.j >= 0) most = o.d2 * (1.f + 1e-6f);
                }
            });
            if (k < n) {
                parent[i] = o.j;
                open[4 * i + 3] = o.und < INFINITY && (o.j < 0 || !(o.und > o.d2 * (1.f + 1e-6f)));
            }
        }
        __syncthreads();
        for (int i = tid; i < n; i += NT) {  // the sorted copy is no longer needed
            rho64[i] = 0.0;
            if (need[i] >> 24) root[atomicAdd(&n_list, 1)] = i;
            need[i] = 0;
        }
        __syncthreads();
        const int listed = n_list;
        if (listed > 0) {
            // a warp per listed row: marks the points to be known in FP64
            for (int e = w; e < listed; e += NT / 32) {
                const int i = root[e];
                RqsBest o = {parent[i], 0.f, 0.f};
                if (o.j >= 0) o.d2 = dist2f(pts[i], pts[o.j]);
                rqs_row<RQS_MARK>(rp, i, o);
            }
            __syncthreads();
            // their FP64 densities, by all threads, summed in any order; terms
            // below e^-41 (at most 4096 of them, of a sum of 1 or more) left out
            const float inv2s2 = (float)a.inv2s2;
            int before = 0, *list = csize;
            for (int b0 = 0; b0 < n; b0 += 32)
                for (unsigned m = __ballot_sync(0xffffffffu, b0 + lane < n && need[b0 + lane]); m; m &= m - 1) {
                    const int i = b0 + __ffs(m) - 1;
                    const float4 p = pts[i];
                    for (int j = tid; j < n; j += NT)
                        if (!(dist2f(p, pts[j]) * inv2s2 > 41.f)) list[atomicAdd(&n_near, 1) - before] = j;
                    __syncthreads();
                    const int end = n_near, c = end - before;
                    before = end;
                    if (w * 32 < c) {
                        double r = 0.0;
                        for (int e = tid; e < c; e += NT) r += exp(-(dist2(p, pts[list[e]]) * a.inv2s2));
#pragma unroll
                        for (int off = 16; off > 0; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
                        if (lane == 0) atomicAdd(&rho64[i], r);
                    }
                    __syncthreads();
                }
            auto again = [&](auto level) {
                for (int e = w; e < listed; e += NT / 32) {
                    RqsBest o;
                    rqs_row<decltype(level)::value>(rp, root[e], o);
                    if (lane == 0) parent[root[e]] = o.j;
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
                            // a term below r 2^-55 leaves r as it is
                            const int j = j0 + lane;
                            const bool adds = j < n && !(dist2f(p, pts[min(j, n - 1)]) * inv2s2 > 38.7f - logf((float)r));
                            if (adds) buf[lane] = exp(-(dist2(p, pts[j]) * a.inv2s2));
                            unsigned m = __ballot_sync(0xffffffffu, adds);
                            __syncwarp();  // the lanes' terms are read by all (a vote orders no memory)
                            for (; m; m &= m - 1) r += buf[__ffs(m) - 1];
                            __syncwarp();
                        }
                        if (lane == 0) rho64[i0] = r;
                    }
                __syncthreads();
                again(std::integral_constant<int, RQS_ORDER>());
            }
        }
        for (int i = tid; i < n; i += NT) csize[i] = 0;
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
        for (int k = w; k < kept; k += NT / 32) {  // the members of each in index order
            const int r = cl_root[k], c = cl_start[k + 1] - cl_start[k];
            int *mem = order + cl_start[k];
            for (int i0 = 0, f = 0; f < c; i0 += 32) {
                const unsigned in = __ballot_sync(0xffffffffu, i0 + lane < n && root[i0 + lane] == r);
                if (in >> lane & 1u) mem[f + __popc(in & ((1u << lane) - 1u))] = i0 + lane;
                f += __popc(in);
            }
        }
        __syncthreads();
        // Per-cluster statistics, members summed in index order: eight lanes a
        // cluster, which widen and multiply eight members at once; lane o of
        // the eight then carries the o-th running sum.  Four clusters of like
        // size share a warp's FP64 instructions.
        if (w < RQS_STAT_WARPS)
            for (int k0 = 4 * w; k0 < kept; k0 += 4 * RQS_STAT_WARPS) {
                const int o = lane & 7, k = k0 + (lane >> 3);
                const int s0 = k < kept ? cl_start[k] : 0, c = k < kept ? cl_start[k + 1] - s0 : 0;
                const int *mem = order + s0;
                const int most = __shfl_sync(0xffffffffu, c, 0);  // clusters come by descending size
                double *buf = bufs + w * RQS_BUF;
                const double *row = buf + 33 * min(o, 5) + (lane & 24);
                // Sums of FP32 values are exact, so the same in any order, while
                // their bits span at most 53: a lane then adds every eighth.
                double s0x = 0.0, s0y = 0.0, s0z = 0.0;
                Span ex, ey, ez;
                unsigned sr = 0, sg = 0, sb = 0;
                for (int f = o; f < c; f += 8) {
                    const float4 p = pts[mem[f]];
                    s0x += widen(p.x);
                    s0y += widen(p.y);
                    s0z += widen(p.z);
                    ex.add(p.x);
                    ey.add(p.y);
                    ez.add(p.z);
                    const uint32_t rgb = __float_as_uint(p.w);
                    sr += rgb & 255;
                    sg += (rgb >> 8) & 255;
                    sb += (rgb >> 16) & 255;
                }
#pragma unroll
                for (int e = 1; e < 8; e <<= 1) {
                    s0x += __shfl_xor_sync(0xffffffffu, s0x, e);
                    s0y += __shfl_xor_sync(0xffffffffu, s0y, e);
                    s0z += __shfl_xor_sync(0xffffffffu, s0z, e);
                    ex.join(e);
                    ey.join(e);
                    ez.join(e);
                    sr += __shfl_xor_sync(0xffffffffu, sr, e);
                    sg += __shfl_xor_sync(0xffffffffu, sg, e);
                    sb += __shfl_xor_sync(0xffffffffu, sb, e);
                }
                double s = o == 0 ? s0x : o == 1 ? s0y : s0z;
                const bool exact = ex.exact(c) && ey.exact(c) && ez.exact(c);
                if (!__all_sync(0xffffffffu, exact)) {  // one by one
                    double r = 0.0;
                    for (int f = 0; f < most; f += 8) {
                        const int m = c - f;
                        if (o < m) {
                            const float4 p = pts[mem[f + o]];
                            buf[lane] = widen(p.x);
                            buf[33 + lane] = widen(p.y);
                            buf[66 + lane] = widen(p.z);
                        }
                        __syncwarp();
                        if (o < 3)
                            for (int e = 0; e < min(m, 8); ++e) r += row[e];
                        __syncwarp();
                    }
                    if (!exact) s = r;
                }
                const double mean = s / c;
                const double m0 = __shfl_sync(0xffffffffu, mean, lane & 24),
                             m1 = __shfl_sync(0xffffffffu, mean, (lane & 24) + 1),
                             m2 = __shfl_sync(0xffffffffu, mean, (lane & 24) + 2);
                s = 0.0;
                float4 next = o < c ? pts[mem[o]] : make_float4(0.f, 0.f, 0.f, 0.f);
                for (int f = 0; f < most; f += 8) {
                    const int m = c - f;
                    const float4 p = next;
                    if (o < m) {
                        const double e0 = widen(p.x) - m0, e1 = widen(p.y) - m1, e2 = widen(p.z) - m2;
                        buf[lane] = e0 * e0;
                        buf[33 + lane] = e0 * e1;
                        buf[66 + lane] = e0 * e2;
                        buf[99 + lane] = e1 * e1;
                        buf[132 + lane] = e1 * e2;
                        buf[165 + lane] = e2 * e2;
                    }
                    __syncwarp();
                    if (o + 8 < m) next = pts[mem[f + 8 + o]];
                    if (o < 6) {
                        double v[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) v[e] = row[e];
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            if (e < m) s += v[e];
                    }
                    __syncwarp();
                }
                if (k < kept) {
                    if (o < 6) cov[k][o] = c > 1 ? s / (double)(c - 1) : 0.0;
                    if (o < 3) mu[k][o] = mean;
                    if (o == 0) {
                        const size_t e = (size_t)L * a.m_max + k;
                        const unsigned h = (unsigned)c / 2, d = (unsigned)c;
                        a.mrgb[e] = make_uchar4((uint8_t)((sr + h) / d), (uint8_t)((sg + h) / d),
                                                (uint8_t)((sb + h) / d), 0);
                        a.msize[e] = c;
                    }
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
    const size_t K = ((size_t)kappa + 31) / 32 * 32;
    return K * (2 * sizeof(float4) + 2 * sizeof(float) + 2 * sizeof(int)) +
           K / RQS_GROUP * 2 * sizeof(float4) + RQS_STAT_WARPS * RQS_BUF * sizeof(double);
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
