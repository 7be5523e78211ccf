// Scoring kernels of the relocaliser: the energy of Eq. 5 on growing pixel
// sets, cull / halving selection, Levenberg-Marquardt refinement in se(3)
// (Sec. 3.2.3) and model-based ranking by depth raycast (Eq. 6-8).
//
// FP32 arithmetic with fused multiply-adds; FP64 only for poses, the 6x6
// normal-equation solve and the SE(3) update.  Every reduction has a fixed
// shape, so results do not depend on how many frames share a launch.
#include <math.h>

#include <cooperative_groups.h>

#include "internal.h"
#include "relocgb_dev.cuh"
#include "kernels.h"
#include "lm_dev.cuh"

namespace rl {

// ---------------------------------------------------------------------------
// Eq. 5 partial energies.  Block = HT hypotheses of one frame (one per
// thread) x one chunk of the pixel set; the chunk's pixels and their modes
// (decoded to FP32) are staged in shared memory and read by broadcast.
// ---------------------------------------------------------------------------

// Partial energy with S lanes per hypothesis (S a power of two <= 32): lane
// t serves hypothesis h0 + t / S and scans modes t % S, t % S + S, ...  Every
// lane runs every pixel, so the shuffles see the whole warp.
__device__ __noinline__ void energy_split(const EnergyArgs &a, int b, int h0, int nb, int S, int np,
                                          const float4 *s_xc, const float4 *s_m0, const float4 *s_m1,
                                          const float *s_m2, const int *s_cnt) {
    const int hl = threadIdx.x / S, sub = threadIdx.x % S;
    const bool act = hl < nb;
    float r00 = 0.f, r01 = 0.f, r02 = 0.f, t0 = 0.f, r10 = 0.f, r11 = 0.f, r12 = 0.f, t1 = 0.f;
    float r20 = 0.f, r21 = 0.f, r22 = 0.f, t2 = 0.f;
    if (act) {
        const int h = h0 + hl;
        const int id = a.idx ? a.idx[(size_t)b * a.idx_stride + h] : h;
        const double *P = a.pose + ((size_t)b * a.pose_stride + id) * 12;
        r00 = (float)P[0]; r01 = (float)P[1]; r02 = (float)P[2]; t0 = (float)P[3];
        r10 = (float)P[4]; r11 = (float)P[5]; r12 = (float)P[6]; t1 = (float)P[7];
        r20 = (float)P[8]; r21 = (float)P[9]; r22 = (float)P[10]; t2 = (float)P[11];
    }
    float acc = 0.f;
    for (int i = 0; i < np; ++i) {
        const int cnt = s_cnt[i];
        if (cnt == 0) continue;  // the same for every lane
        const float4 x = s_xc[i];
        const float y0 = fmaf(r00, x.x, fmaf(r01, x.y, fmaf(r02, x.z, t0)));
        const float y1 = fmaf(r10, x.x, fmaf(r11, x.y, fmaf(r12, x.z, t1)));
        const float y2 = fmaf(r20, x.x, fmaf(r21, x.y, fmaf(r22, x.z, t2)));
        const int base = i * a.maxm;
        float best = INFINITY;
        if (a.p.use_cov) {
            for (int m = sub; m < cnt; m += S) {
                const float4 m0 = s_m0[base + m], m1 = s_m1[base + m];
                const float u22 = s_m2[base + m];
                const float v0 = y0 - m0.x, v1 = y1 - m0.y, v2 = y2 - m0.z;
                const float w0 = fmaf(m0.w, v0, fmaf(m1.x, v1, m1.y * v2));
                const float w1 = fmaf(m1.z, v1, m1.w * v2);
                const float w2 = u22 * v2;
                best = fminf(best, fmaf(w0, w0, fmaf(w1, w1, w2 * w2)));
            }
        } else {
            for (int m = sub; m < cnt; m += S) {
                const float4 m0 = s_m0[base + m];
                const float v0 = y0 - m0.x, v1 = y1 - m0.y, v2 = y2 - m0.z;
                best = fminf(best, fmaf(v0, v0, fmaf(v1, v1, v2 * v2)));
            }
        }
        for (int off = 1; off < S; off <<= 1) best = fminf(best, __shfl_xor_sync(0xffffffffu, best, off));
        acc += sqrtf(best);
    }
    if (act && sub == 0) a.part[((size_t)b * a.part_h + h0 + hl) * a.n_chunks + blockIdx.y] = acc;
}

__global__ void __launch_bounds__(256) k_energy(EnergyArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    float4 *s_xc = (float4 *)smem;                         // [chunk]
    float4 *s_m0 = s_xc + a.chunk;                         // [chunk*maxm] mu.xyz, U00
    float4 *s_m1 = s_m0 + a.chunk * a.maxm;                // [chunk*maxm] U01 U02 U11 U12
    float *s_m2 = (float *)(s_m1 + a.chunk * a.maxm);      // [chunk*maxm] U22
    int *s_cnt = (int *)(s_m2 + a.chunk * a.maxm);         // [chunk]

    const int b = blockIdx.z;
    const int n = a.count[b];
    if (a.round_gate && !round_active(n, a.p)) return;
    const int h0 = blockIdx.x * blockDim.x;
    if (h0 >= n) return;
    const int p0 = blockIdx.y * a.chunk;
    if (p0 >= a.n_pix) return;
    const int np = min(a.chunk, a.n_pix - p0);
    const float4 *xc = a.xc + (size_t)b * a.max_pix + p0;
    const size_t row0 = (size_t)b * a.max_pix + p0;   // first table row of the chunk
    for (int i = threadIdx.x; i < np; i += blockDim.x) {
        s_xc[i] = xc[i];
        s_cnt[i] = a.q_tab_cnt[row0 + i];
    }
    // the chunk's rows of the mode table are contiguous: coalesced copy
    const int mpad = a.p.mpad;
    const float4 *tb0 = a.q_tab0 + row0 * mpad;
    const float4 *tb1 = a.q_tab1 + row0 * mpad;
    const float *tb2 = a.q_tab2 + row0 * mpad;
    for (int e = threadIdx.x; e < np * mpad; e += blockDim.x) {
        s_m0[e] = tb0[e];
        if (a.p.use_cov) {
            s_m1[e] = tb1[e];
            s_m2[e] = tb2[e];
        }
    }
    __syncthreads();
    if (a.work && threadIdx.x == 0) {
        unsigned long long pairs = 0, modes = 0;
        for (int i = 0; i < np; ++i)
            if (s_cnt[i] > 0) {
                ++pairs;
                modes += (unsigned long long)s_cnt[i];
            }
        const unsigned long long nh = (unsigned long long)min((int)blockDim.x, n - h0);
        atomicAdd(&a.work[W_E_PAIRS], nh * pairs);
        atomicAdd(&a.work[W_E_MODES], nh * modes);
    }
    // With fewer hypotheses than threads, S adjacent lanes share one and
    // split each pixel's mode scan (every S-th mode); the minimum is exact in
    // any order, so the partial energy is the same as with one lane.
    const int nb = min((int)blockDim.x, n - h0);
    int hb = 1;
    while (hb < nb) hb <<= 1;
    const int S = min(32, (int)blockDim.x / hb);
    if (S > 1) {
        energy_split(a, b, h0, nb, S, np, s_xc, s_m0, s_m1, s_m2, s_cnt);
        return;
    }
    const int h = h0 + threadIdx.x;
    if (h >= n) return;
    const int id = a.idx ? a.idx[(size_t)b * a.idx_stride + h] : h;
    const double *P = a.pose + ((size_t)b * a.pose_stride + id) * 12;
    const float r00 = (float)P[0], r01 = (float)P[1], r02 = (float)P[2], t0 = (float)P[3];
    const float r10 = (float)P[4], r11 = (float)P[5], r12 = (float)P[6], t1 = (float)P[7];
    const float r20 = (float)P[8], r21 = (float)P[9], r22 = (float)P[10], t2 = (float)P[11];
    float acc = 0.f;
    for (int i = 0; i < np; ++i) {
        const int cnt = s_cnt[i];
        if (cnt == 0) continue;
        const float4 x = s_xc[i];
        const float y0 = fmaf(r00, x.x, fmaf(r01, x.y, fmaf(r02, x.z, t0)));
        const float y1 = fmaf(r10, x.x, fmaf(r11, x.y, fmaf(r12, x.z, t1)));
        const float y2 = fmaf(r20, x.x, fmaf(r21, x.y, fmaf(r22, x.z, t2)));
        const int base = i * a.maxm;
        float best = INFINITY;
        if (a.p.use_cov) {
            for (int m = 0; m < cnt; ++m) {
                const float4 m0 = s_m0[base + m], m1 = s_m1[base + m];
                const float u22 = s_m2[base + m];
                const float v0 = y0 - m0.x, v1 = y1 - m0.y, v2 = y2 - m0.z;
                const float w0 = fmaf(m0.w, v0, fmaf(m1.x, v1, m1.y * v2));
                const float w1 = fmaf(m1.z, v1, m1.w * v2);
                const float w2 = u22 * v2;
                best = fminf(best, fmaf(w0, w0, fmaf(w1, w1, w2 * w2)));
            }
        } else {
            for (int m = 0; m < cnt; ++m) {
                const float4 m0 = s_m0[base + m];
                const float v0 = y0 - m0.x, v1 = y1 - m0.y, v2 = y2 - m0.z;
                best = fminf(best, fmaf(v0, v0, fmaf(v1, v1, v2 * v2)));
            }
        }
        acc += sqrtf(best);
    }
    a.part[((size_t)b * a.part_h + h) * a.n_chunks + blockIdx.y] = acc;
}

// ---------------------------------------------------------------------------
// Cull (phase 0) and halving rounds (phase 1): sum the partial energies in
// chunk order, rank by (E, slot), keep the best min(n, N_cull) or ceil(n/2).
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(1024) k_select(SelectArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ float s_tile[64][33];
    float *sE = (float *)smem;                       // [n]
    int *sS = (int *)(sE + a.p.n_hyp);               // [n]
    double *sP = (double *)(sS + a.p.n_hyp);         // [n_cull][12]
    float *sKE = (float *)(sP + a.p.n_cull * 12);    // [n_cull]
    int *sKS = (int *)(sKE + a.p.n_cull);            // [n_cull]
    const int b = blockIdx.x, tid = threadIdx.x;
    const int n = a.count[b];
    if (a.phase == 1 && !round_active(n, a.p)) return;
    const int N = a.p.n_hyp, NC = a.p.n_cull;
    const bool from_parts = !(a.phase == 1 && a.energy_from_lm);
    // Long rows of partial energies (modes too many for 32 pixels a chunk) are
    // read by the whole block, 64 rows by 32 chunks at a time and the next
    // tile's loads in flight, and summed in chunk order from shared memory: a
    // thread walking its own row of 125 to 875 chunks took 30 to 75 us.
    // Shorter rows are a line or two, read directly.
    const bool tiled = from_parts && a.n_chunks_used > 64;
    if (tiled) {
        const int nct = (a.n_chunks_used + 31) / 32, nt = (n + 63) / 64 * nct;
        const int r0 = tid >> 5, c0 = tid & 31;
        auto part = [&](int tile, int r) {
            const int h = tile / nct * 64 + r, c = tile % nct * 32 + c0;
            return tile < nt && h < n && c < a.n_chunks_used ? a.part[((size_t)b * a.part_h + h) * a.n_chunks + c] : 0.f;
        };
        float e = 0.f, p0 = part(0, r0), p1 = part(0, r0 + 32);
        for (int tile = 0; tile < nt; ++tile) {
            s_tile[r0][c0] = p0;
            s_tile[r0 + 32][c0] = p1;
            p0 = part(tile + 1, r0);
            p1 = part(tile + 1, r0 + 32);
            __syncthreads();
            const int h = tile / nct * 64 + tid, cb = tile % nct * 32;
            if (tid < 64 && h < n) {
                const int m = min(32, a.n_chunks_used - cb);
                for (int c = 0; c < m; ++c) e += s_tile[tid][c];
                if (tile % nct == nct - 1) {
                    sE[h] = e;
                    e = 0.f;
                }
            }
            __syncthreads();
        }
    }
    for (int i = tid; i < n; i += blockDim.x) {
        float e = 0.f;
        if (!from_parts) {
            e = a.q.cur_energy[(size_t)b * NC + i];
        } else if (tiled) {
            e = sE[i];
        } else {
            const float *pp = a.part + ((size_t)b * a.part_h + i) * a.n_chunks;
            for (int c = 0; c < a.n_chunks_used; ++c) e += pp[c];
        }
        if (isnan(e)) e = INFINITY;
        sE[i] = e;
        sS[i] = a.phase == 0 ? a.hyp_list[(size_t)b * N + i] : a.q.cur_slot[(size_t)b * NC + i];
    }
    __syncthreads();
    const int keep = a.phase == 0 ? min(n, NC) : (n + 1) / 2;
    for (int i = tid; i < n; i += blockDim.x) {
        const float e = sE[i];
        const int s = sS[i];
        int rank = 0;
        for (int j = 0; j < n; ++j) {
            const float f = sE[j];
            rank += (f < e) || (f == e && sS[j] < s);
        }
        if (rank < keep) {
            const double *src = a.phase == 0 ? a.hyp_pose + ((size_t)b * N + s) * 12
                                             : a.q.cur_pose + ((size_t)b * NC + i) * 12;
            for (int k = 0; k < 12; ++k) sP[rank * 12 + k] = src[k];
            sKE[rank] = e;
            sKS[rank] = s;
        }
    }
    __syncthreads();
    for (int i = tid; i < keep; i += blockDim.x) {
        for (int k = 0; k < 12; ++k) a.q.cur_pose[((size_t)b * NC + i) * 12 + k] = sP[i * 12 + k];
        a.q.cur_energy[(size_t)b * NC + i] = sKE[i];
        a.q.cur_slot[(size_t)b * NC + i] = sKS[i];
    }
    if (a.phase == 0)
        for (int i = tid; i < keep; i += blockDim.x) {
            a.q.cull_slot[(size_t)b * NC + i] = sKS[i];
            a.q.cull_energy[(size_t)b * NC + i] = sKE[i];
        }
    const bool take = a.q.n_chosen[b] < 0 && keep <= a.p.k_out;
    if (take)
        for (int i = tid; i < keep; i += blockDim.x) {
            for (int k = 0; k < 12; ++k)
                a.q.chosen_pose[((size_t)b * 16 + i) * 12 + k] = sP[i * 12 + k];
            a.q.chosen_energy[(size_t)b * 16 + i] = sKE[i];
            a.q.chosen_slot[(size_t)b * 16 + i] = sKS[i];
        }
    if (a.phase == 1 && a.round < 16)
        for (int i = tid; i < keep; i += blockDim.x) {
            const size_t o = ((size_t)b * 16 + a.round) * NC + i;
            a.q.round_slot[o] = sKS[i];
            a.q.round_energy[o] = sKE[i];
            for (int k = 0; k < 12; ++k) a.q.round_pose[o * 12 + k] = sP[i * 12 + k];
        }
    __syncthreads();
    if (tid == 0) {
        a.q.n_cur[b] = keep;
        a.q.n_pix[b] = a.n_pix;
        if (take) {
            a.q.n_chosen[b] = keep;
            a.q.chosen_npix[b] = a.n_pix;
        }
        if (a.phase == 1) {
            if (a.round < 16) a.q.round_count[(size_t)b * 16 + a.round] = keep;
            a.q.n_rounds[b] = a.round + 1;
        }
    }
}

// ---------------------------------------------------------------------------
// Levenberg-Marquardt in se(3) (Sec. 3.2.3) for rows of the mode table too
// long for the cluster kernel's staged tiles (lm.cu).
// ---------------------------------------------------------------------------

// LM, hypotheses spread over threads.  A round's n hypotheses of a frame are
// split over up to LM3_BPQ parts; inside a part, hypothesis h has G = 256 / HB
// pixel groups (HB = the next power of two >= the part's hypothesis count),
// group g taking the pixels g, g + G, ...  As rounds halve n, each hypothesis
// gets more groups.  Partial normal equations are tree-reduced over the
// groups (fixed shape), the 6x6 system of each hypothesis is solved in FP64
// by one thread, and the trial cost with the same correspondences is reduced
// the same way.
//
// A part is one cluster of CT blocks: block c takes the groups c, c + CT, ...,
// and CT adjacent lanes share a pair's mode scan (every CT-th mode; ties to
// the lower index), so the sums and their order do not depend on CT.  The
// tree's levels of at least CT groups apart lie within a block, the last ones
// go through distributed shared memory, every block holding the same totals
// and taking the same decisions.  With one block per part a call of few
// frames leaves most of the GPU idle (four frames: 16 blocks) on scans of up
// to 250 modes; CT grows to 8 while the call's blocks still fit two per SM.
// A large batch keeps CT = 1: the lanes that share a scan idle through the
// accumulation, about a quarter more instructions.  Measured on four 640x480
// frames, 64 hypotheses, up to 250 modes per pixel, six rounds: 4.2 ms with
// CT = 8 (4.4 when a step's count and point were not loaded a step ahead),
// 17.9 with one block per part.  What bounds it then is the latency of a
// step's chain of loads with two warps per sub-partition, not the scan:
// CT = 16 took as long, and so did rows read once for a warp's hypotheses
// (4.8 ms) or eight modes at a time (5.2 ms).
constexpr int LM3_THREADS = 256;
constexpr int LM3_BPQ = 4;
constexpr int LM3_HMAX = 64 / LM3_BPQ;  // hypotheses of a part (n_cull <= 64)
constexpr int LM3_NV = 29;              // 21 J^T J, 6 J^T r, cost, inliers

template <int CT>
__global__ void __launch_bounds__(LM3_THREADS, 2) k_lm_spread(LmArgs a) {
    constexpr int PAIRS = LM3_THREADS / CT;           // (hypothesis, group) pairs of a block
    __shared__ float s_red[PAIRS * (LM3_NV + 4)];     // partial sums of each pair
    __shared__ float s_trial[PAIRS];
    __shared__ double s_H[LM3_HMAX][12];              // current pose per hypothesis of the part
    __shared__ double s_Hn[LM3_HMAX][12];             // trial pose
    __shared__ double s_lambda[LM3_HMAX];
    __shared__ float s_tot[LM3_HMAX][LM3_NV];
    __shared__ int s_state[LM3_HMAX];                 // 1 active, 0 stopped
    constexpr int RS = LM3_NV + 4;                    // odd row stride
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int rank = CT > 1 ? (int)cluster.block_rank() : 0;
    const int b = blockIdx.y;
    const int n = a.q.n_cur[b];
    if (!round_active(n, a.p)) return;
    // hypotheses of this part: [h0, h0 + nb)
    const int per = (n + LM3_BPQ - 1) / LM3_BPQ;
    const int h0 = (int)(blockIdx.x / CT) * per;
    const int nb = min(per, n - h0);
    if (nb <= 0) return;
    int HB = 1;
    while (HB < nb) HB <<= 1;
    const int G = LM3_THREADS / HB, GL = G / CT;      // groups, and those of this block
    const int t = threadIdx.x, sub = t % CT, pair = t / CT;
    const int hl = pair % HB, g = pair / HB * CT + rank;
    const bool mine = hl < nb;
    const int NC = a.p.n_cull;
    const size_t row0 = (size_t)b * a.p.max_pix;
    const int stride = a.p.mpad;
    const float4 *xcs = a.q.xc + row0;
    const float4 *t0 = a.q.tab0 + row0 * stride;
    const float4 *t1 = a.q.tab1 + row0 * stride;
    const float *t2 = a.q.tab2 + row0 * stride;
    const int16_t *tcnt = a.q.tab_cnt + row0;
    // correspondences [pixel][nb] of the part's hypotheses (local mode index, -1 none)
    int32_t *corr = a.q.corr + ((size_t)b * NC + h0) * a.p.max_pix;
    const float thr2 = (float)(a.p.lm_inlier_thresh * a.p.lm_inlier_thresh);
    const bool cov = a.p.use_cov;
    for (int i = t; i < nb * 12; i += LM3_THREADS) s_H[i / 12][i % 12] = a.q.cur_pose[((size_t)b * NC + h0 + i / 12) * 12 + i % 12];
    for (int i = t; i < nb; i += LM3_THREADS) {
        s_lambda[i] = a.p.lm_lambda0;
        s_state[i] = 1;
    }
    __syncthreads();
    // Tree sum over the groups of value k of row `stride_` arrays in `part`
    // (left in the rows of local group 0), then over the cluster; f(h, k, sum).
    auto reduce = [&](float *part, int nv, int rs, auto f) {
        __syncthreads();
        for (int s = GL >> 1; s > 0; s >>= 1) {
            for (int e = t; e < s * HB * nv; e += LM3_THREADS)
                part[e / nv * rs + e % nv] += part[(e / nv + s * HB) * rs + e % nv];
            __syncthreads();
        }
        if (CT > 1) cluster.sync();
        for (int e = t; e < nb * nv; e += LM3_THREADS) {
            const int h = e / nv, k = e % nv;
            float v[CT];
#pragma unroll
            for (int r = 0; r < CT; ++r) v[r] = (CT > 1 ? cluster.map_shared_rank(part, r) : part)[h * rs + k];
#pragma unroll
            for (int s = CT / 2; s > 0; s >>= 1)
#pragma unroll
                for (int r = 0; r < s; ++r) v[r] += v[r + s];
            f(h, k, v[0]);
        }
        __syncthreads();
    };
    const int steps = (a.n_pix + G - 1) / G;  // pixels of a group, the same for every lane
    unsigned w_pairs = 0, w_modes = 0, w_in = 0, w_trial = 0;
    for (int it = 0; it < a.p.lm_max_iter; ++it) {
        const bool act = mine && s_state[hl];
        if (!__syncthreads_or(act)) break;  // the same in every block of the cluster
        float acc[28];
#pragma unroll
        for (int k = 0; k < 28; ++k) acc[k] = 0.f;
        int nin = 0;
        {
            float P[12];
#pragma unroll
            for (int k = 0; k < 12; ++k) P[k] = act ? (float)s_H[hl][k] : 0.f;
            int next_cnt = 0;
            float4 next_x = make_float4(0.f, 0.f, 0.f, 0.f);
            auto fetch = [&](int st) {  // a step ahead: what its scan waits for
                const int i = st * G + g;
                const bool on = act && i < a.n_pix;
                next_cnt = on ? (int)tcnt[i] : 0;
                if (on) next_x = xcs[i];
            };
            fetch(0);
            for (int st = 0; st < steps; ++st) {
                const int i = st * G + g;
                const bool on = act && i < a.n_pix;
                const int cnt = next_cnt;
                const float4 x = next_x;
                fetch(st + 1);
                const size_t base = (size_t)i * stride;
                float y0 = 0.f, y1 = 0.f, y2 = 0.f;
                if (cnt > 0) {
                    y0 = fmaf(P[0], x.x, fmaf(P[1], x.y, fmaf(P[2], x.z, P[3])));
                    y1 = fmaf(P[4], x.x, fmaf(P[5], x.y, fmaf(P[6], x.z, P[7])));
                    y2 = fmaf(P[8], x.x, fmaf(P[9], x.y, fmaf(P[10], x.z, P[11])));
                }
                float best = INFINITY;
                int best_m = -1;
                if (cov) {
#pragma unroll 4
                    for (int m = sub; m < cnt; m += CT) {
                        const float4 m0 = __ldg(&t0[base + m]), m1 = __ldg(&t1[base + m]);
                        const float u22 = __ldg(&t2[base + m]);
                        const float v0 = y0 - m0.x, v1 = y1 - m0.y, v2 = y2 - m0.z;
                        const float w0 = fmaf(m0.w, v0, fmaf(m1.x, v1, m1.y * v2));
                        const float w1 = fmaf(m1.z, v1, m1.w * v2);
                        const float w2 = u22 * v2;
                        const float d2 = fmaf(w0, w0, fmaf(w1, w1, w2 * w2));
                        if (d2 < best) {
                            best = d2;
                            best_m = m;
                        }
                    }
                } else {
#pragma unroll 4
                    for (int m = sub; m < cnt; m += CT) {
                        const float4 m0 = __ldg(&t0[base + m]);
                        const float v0 = y0 - m0.x, v1 = y1 - m0.y, v2 = y2 - m0.z;
                        const float d2 = fmaf(v0, v0, fmaf(v1, v1, v2 * v2));
                        if (d2 < best) {
                            best = d2;
                            best_m = m;
                        }
                    }
                }
#pragma unroll
                for (int off = 1; off < CT; off <<= 1) {
                    const float ob = __shfl_xor_sync(0xffffffffu, best, off);
                    const int om = __shfl_xor_sync(0xffffffffu, best_m, off);
                    if (om >= 0 && (best_m < 0 || ob < best || (ob == best && om < best_m))) {
                        best = ob;
                        best_m = om;
                    }
                }
                if (!on || sub != 0) continue;
                if (cnt > 0) {
                    ++w_pairs;
                    w_modes += cnt;
                }
                if (best_m >= 0) {
                    const float4 m0 = __ldg(&t0[base + best_m]);
                    const float v0 = y0 - m0.x, v1 = y1 - m0.y, v2 = y2 - m0.z;
                    if (fmaf(v0, v0, fmaf(v1, v1, v2 * v2)) <= thr2) {
                        ++nin;
                        ++w_in;
                        if (cov) {
                            const float4 m1 = __ldg(&t1[base + best_m]);
                            lm_accumulate(y0, y1, y2, v0, v1, v2, m0.w, m1.x, m1.y, m1.z, m1.w,
                                           __ldg(&t2[base + best_m]), acc);
                        } else {
                            lm_accumulate(y0, y1, y2, v0, v1, v2, 1.f, 0.f, 0.f, 1.f, 0.f, 1.f, acc);
                        }
                    } else {
                        best_m = -1;
                    }
                }
                corr[(size_t)i * nb + hl] = best_m;
            }
        }
        if (sub == 0) {
#pragma unroll
            for (int k = 0; k < 28; ++k) s_red[pair * RS + k] = acc[k];
            s_red[pair * RS + 28] = (float)nin;
        }
        reduce(s_red, LM3_NV, RS, [&](int h, int k, float v) { s_tot[h][k] = v; });
        // FP64 solve per active hypothesis
        if (t < nb && s_state[t]) {
            int status = s_tot[t][28] < 3.f ? 1 : 0;
            double step[6];
            if (!status) {
                double A[36], rhs[6];
                int k = 0;
                for (int r = 0; r < 6; ++r)
                    for (int c = r; c < 6; ++c, ++k) A[6 * r + c] = A[6 * c + r] = (double)s_tot[t][k];
                for (int r = 0; r < 6; ++r) {
                    A[6 * r + r] += s_lambda[t] * (double)s_tot[t][r * 6 - r * (r - 1) / 2];
                    rhs[r] = -(double)s_tot[t][21 + r];
                }
                if (!chol_solve6(A, rhs, step)) {
                    status = 1;
                } else {
                    double sn = 0.0;
                    for (int r = 0; r < 6; ++r) sn += step[r] * step[r];
                    if (sqrt(sn) < a.p.lm_stop) status = 1;
                }
            }
            if (status) {
                s_state[t] = 0;
            } else {
                double Hn[12];
                for (int i = 0; i < 12; ++i) Hn[i] = s_H[t][i];
                se3_left(step, Hn);
                for (int i = 0; i < 12; ++i) s_Hn[t][i] = Hn[i];
            }
        }
        __syncthreads();
        // Trial cost with the same correspondences.  The CT lanes of a pair
        // take a pixel each, their residuals are added in pixel order.
        const bool act2 = mine && s_state[hl];
        float trial = 0.f;
        {
            float P[12];
#pragma unroll
            for (int k = 0; k < 12; ++k) P[k] = act2 ? (float)s_Hn[hl][k] : 0.f;
            for (int st = 0; st < steps; st += CT) {
                const int i = (st + sub) * G + g;
                const int m = act2 && i < a.n_pix ? corr[(size_t)i * nb + hl] : -1;
                float r0 = 0.f, r1 = 0.f, r2 = 0.f;
                if (m >= 0) {
                    ++w_trial;
                    const float4 x = xcs[i];
                    const size_t e = (size_t)i * stride + m;
                    const float4 m0 = __ldg(&t0[e]);
                    const float y0 = fmaf(P[0], x.x, fmaf(P[1], x.y, fmaf(P[2], x.z, P[3])));
                    const float y1 = fmaf(P[4], x.x, fmaf(P[5], x.y, fmaf(P[6], x.z, P[7])));
                    const float y2 = fmaf(P[8], x.x, fmaf(P[9], x.y, fmaf(P[10], x.z, P[11])));
                    const float v0 = y0 - m0.x, v1 = y1 - m0.y, v2 = y2 - m0.z;
                    if (cov) {
                        const float4 m1 = __ldg(&t1[e]);
                        r0 = fmaf(m0.w, v0, fmaf(m1.x, v1, m1.y * v2));
                        r1 = fmaf(m1.z, v1, m1.w * v2);
                        r2 = __ldg(&t2[e]) * v2;
                    } else {
                        r0 = v0;
                        r1 = v1;
                        r2 = v2;
                    }
                }
#pragma unroll
                for (int k = 0; k < CT; ++k) {
                    const float q0 = __shfl_sync(0xffffffffu, r0, k, CT), q1 = __shfl_sync(0xffffffffu, r1, k, CT),
                                q2 = __shfl_sync(0xffffffffu, r2, k, CT);
                    trial = fmaf(q0, q0, fmaf(q1, q1, fmaf(q2, q2, trial)));  // + 0 where there is none
                }
            }
        }
        if (sub == 0) s_trial[pair] = trial;
        reduce(s_trial, 1, 1, [&](int h, int, float v) {
            if (!s_state[h]) return;
            if (v < s_tot[h][27]) {
                for (int i = 0; i < 12; ++i) s_H[h][i] = s_Hn[h][i];
                s_lambda[h] /= 10.0;
            } else {
                s_lambda[h] *= 10.0;
            }
        });
    }
    if (rank == 0)
        for (int i = t; i < nb * 12; i += LM3_THREADS)
            a.q.cur_pose[((size_t)b * NC + h0 + i / 12) * 12 + i % 12] = s_H[i / 12][i % 12];
    if (a.work && (w_pairs | w_trial)) {
        atomicAdd(&a.work[W_LM_PAIRS], (unsigned long long)w_pairs);
        atomicAdd(&a.work[W_LM_MODES], (unsigned long long)w_modes);
        atomicAdd(&a.work[W_LM_INLIERS], (unsigned long long)w_in);
        atomicAdd(&a.work[W_LM_TRIAL], (unsigned long long)w_trial);
    }
    if (CT > 1) cluster.sync();  // no block leaves while another may still read its shared memory
}

template <int CT>
static rl_status launch_lm_spread(const LmArgs &a, int n, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(LM3_BPQ * CT, n);
    cfg.blockDim = dim3(LM3_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = CT;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    RL_CK(cudaLaunchKernelEx(&cfg, k_lm_spread<CT>, a));
    return RL_OK;
}

// z-depth of the first box face hit by the ray of pixel (u, v) (exit point
// from inside the box, entry point from outside), in FP64.
__device__ bool ray_depth64(const double *P, int u, int v, float fx, float fy, float cx, float cy,
                            const double lo[3], const double hi[3], double *depth) {
    const double dc0 = ((double)u - (double)cx) / (double)fx;
    const double dc1 = ((double)v - (double)cy) / (double)fy;
    double tn = -INFINITY, tf = INFINITY;
    for (int ax = 0; ax < 3; ++ax) {
        const double d = P[4 * ax] * dc0 + P[4 * ax + 1] * dc1 + P[4 * ax + 2];
        const double o = P[4 * ax + 3];
        if (d == 0.0) {
            if (o < lo[ax] || o > hi[ax]) return false;
            continue;
        }
        const double t1 = (lo[ax] - o) / d, t2 = (hi[ax] - o) / d;
        tn = fmax(tn, fmin(t1, t2));
        tf = fmin(tf, fmax(t1, t2));
    }
    if (tn > tf) return false;
    if (tn > 0.0) { *depth = tn; return true; }
    if (tf > 0.0) { *depth = tf; return true; }
    return false;
}

// The FP64 re-evaluation of one ray, kept out of line so that none of its
// FP64 work is scheduled into the FP32 loop that rarely needs it.
__device__ __noinline__ bool ray_depth_fp64(const double *P, int u, int v, float fx, float fy, float cx, float cy,
                                            const double lo[3], const double hi[3], float *depth) {
    double dd = 0.0;
    const bool ok = ray_depth64(P, u, v, fx, fy, cx, cy, lo, hi, &dd);
    *depth = (float)dd;
    return ok;
}

// One ray of a camera inside or outside the box against the general slab
// test: *depth of the first face hit, false when there is none.  A decision
// within a relative margin of 1e-4 of changing is taken in FP64 (n64 counts
// them).
__device__ __noinline__ bool ray_depth_slab(const RaycastArgs &a, const Frame &fr, const float *P, const double *P64,
                                            float dc0, float dc1, int u, int v, float *depth, unsigned &n64) {
    float d[3], o[3];
    for (int r = 0; r < 3; ++r) {
        d[r] = fmaf(P[4 * r], dc0, fmaf(P[4 * r + 1], dc1, P[4 * r + 2]));
        o[r] = P[4 * r + 3];
    }
    const float dn = fabsf(d[0]) + fabsf(d[1]) + fabsf(d[2]);
    float tn = -INFINITY, tf = INFINITY;
    bool unsure = false;
    for (int ax = 0; ax < 3; ++ax) {
        if (fabsf(d[ax]) <= 1e-5f * dn) {
            unsure = true;
            continue;
        }
        const float inv = __fdividef(1.0f, d[ax]);
        const float ta = (a.lo[ax] - o[ax]) * inv, tb = (a.hi[ax] - o[ax]) * inv;
        tn = fmaxf(tn, fminf(ta, tb));
        tf = fminf(tf, fmaxf(ta, tb));
    }
    if (!unsure) {
        const float scale = fmaxf(fabsf(tn), fabsf(tf));
        if (fabsf(tf - tn) <= 1e-4f * scale || fabsf(tn) <= 1e-4f * scale || fabsf(tf) <= 1e-4f * scale) unsure = true;
    }
    if (unsure) {
        ++n64;
        return ray_depth_fp64(P64, u, v, fr.fx, fr.fy, fr.cx, fr.cy, a.lo64, a.hi64, depth);
    }
    if (tn <= tf && tn > 0.f) {
        *depth = tn;
        return true;
    }
    if (tn <= tf && tf > 0.f) {
        *depth = tf;
        return true;
    }
    return false;
}

// Each thread owns RC_PIX pixels of an RC_TILE-pixel tile and runs all poses
// of the frame over them in turn (poses staged in shared memory, RC_CHUNK at a
// time), so each pixel's live depth and viewing direction are read once.
//
// A camera more than 1 mm inside the box: every ray leaves the box exactly
// once, at the nearest exit plane; with t_ax = (bound - o) / d, bound = hi
// for d >= +0 and lo for d <= -0 (a zero component then gives +inf), the
// depth is min_ax t_ax, a continuous function of the ray with no hit/miss
// decision to certify.  The approximate reciprocal maps +-0 to +-inf.  Other
// cameras take the slab test.
//
// Per pose the tile's sums are reduced over the thread's pixels in order,
// then over lanes (l + l' at distance 16, 8, 4, 2, 1), then over warps in
// order, one partial per (pose, tile).  While every pose of a chunk is inside
// the box, four poses' sums are reduced over the lanes together, the first
// two steps halving the poses a lane carries: 6 shuffles for 4 poses instead
// of 20; the counts of rays and of live pixels are then the same for every
// pose.  (All 16 poses of a chunk at once take fewer shuffles still, but
// their straight-line code is fetched cold by every block of a call of few
// frames: one frame's ranking 31 us instead of 27.)  What bounds it is issue
// (78% of cycles) and the ALU.  Measured at 640x480: 128 poses of a frame 49
// us (109 with the sums of one pose reduced at a time and rescaling
// divisions), 16 poses of 8 frames 78 us (90 to 101), of one frame 27 (25).
constexpr int RC_CHUNK = 16, RC_GROUP = 4;
static_assert(RC_GROUP == 4 && RC_CHUNK % RC_GROUP == 0, "the lanes' pose index takes bits 4 and 3");

__global__ void __launch_bounds__(256, 4) k_raycast_score(RaycastArgs a) {
    __shared__ __align__(16) float sPf[RC_CHUNK][12];
    __shared__ __align__(16) float s_exit[RC_CHUNK][8];  // lo - o, hi - o per axis (x, y, z, -)
    __shared__ float s_sum[RC_CHUNK][8];
    __shared__ int s_syn[RC_CHUNK][8], s_both[RC_CHUNK][8];
    const int b = blockIdx.y;
    const int n_poses = a.n_poses_of(b);
    if (n_poses <= 0) return;
    const Frame fr = a.frames[b];
    const int npx = fr.W * fr.H;
    int u[RC_PIX], v[RC_PIX];
    float dc0[RC_PIX], dc1[RC_PIX], dl[RC_PIX];
    bool in[RC_PIX];
#pragma unroll
    for (int q = 0; q < RC_PIX; ++q) {
        const int p = blockIdx.x * RC_TILE + q * 256 + threadIdx.x;
        in[q] = p < npx;
        u[q] = 0; v[q] = 0;
        dc0[q] = 0.f; dc1[q] = 0.f; dl[q] = 0.f;
        if (in[q]) {
            u[q] = p % fr.W;
            v[q] = p / fr.W;
            // fast approximate divisions: their few-ulp error is far inside
            // the margin that sends a ray to the FP64 path
            dc0[q] = __fdividef((float)u[q] - fr.cx, fr.fx);
            dc1[q] = __fdividef((float)v[q] - fr.cy, fr.fy);
            dl[q] = fr.depth[p];
        }
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int n_in = 0, n_live = 0;  // this thread's pixels, and those with depth
#pragma unroll
    for (int q = 0; q < RC_PIX; ++q) {
        n_in += in[q];
        n_live += in[q] && dl[q] > 0.f;
    }
    const int w_in = __reduce_add_sync(0xffffffffu, n_in), w_live = __reduce_add_sync(0xffffffffu, n_live);
    unsigned n64 = 0;  // rays re-evaluated in FP64 (profiling counter)
    for (int c0 = 0; c0 < n_poses; c0 += RC_CHUNK) {
        const int cnt = min(RC_CHUNK, n_poses - c0);
        __syncthreads();  // the previous chunk's poses and partials are consumed
        // poses past the last repeat it; their sums are dropped
        for (int e = threadIdx.x; e < RC_CHUNK * 12; e += blockDim.x)
            sPf[e / 12][e % 12] = (float)a.pose_of(b, c0 + min(e / 12, cnt - 1))[e % 12];
        __syncthreads();
        bool inside = true;
        if (threadIdx.x < RC_CHUNK) {
            const float *P = sPf[threadIdx.x];
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                const float o = P[4 * ax + 3];
                inside = inside && o - a.lo[ax] > 1e-3f && a.hi[ax] - o > 1e-3f;
                s_exit[threadIdx.x][ax] = a.lo[ax] - o;
                s_exit[threadIdx.x][4 + ax] = a.hi[ax] - o;
            }
        }
        if (__syncthreads_and(inside)) {
#pragma unroll 1
            for (int g = 0; g < cnt; g += RC_GROUP) {
                float sum[RC_GROUP];
#pragma unroll
                for (int k = 0; k < RC_GROUP; ++k) {
                    const float4 P0 = *(const float4 *)&sPf[g + k][0], P1 = *(const float4 *)&sPf[g + k][4],
                                 P2 = *(const float4 *)&sPf[g + k][8];
                    const float4 lo = *(const float4 *)&s_exit[g + k][0], hi = *(const float4 *)&s_exit[g + k][4];
                    sum[k] = 0.f;
#pragma unroll
                    for (int q = 0; q < RC_PIX; ++q) {
                        const float d0 = fmaf(P0.x, dc0[q], fmaf(P0.y, dc1[q], P0.z));
                        const float d1 = fmaf(P1.x, dc0[q], fmaf(P1.y, dc1[q], P1.z));
                        const float d2 = fmaf(P2.x, dc0[q], fmaf(P2.y, dc1[q], P2.z));
                        const float t0 = (signbit(d0) ? lo.x : hi.x) * rcp_approx(d0);
                        const float t1 = (signbit(d1) ? lo.y : hi.y) * rcp_approx(d1);
                        const float t2 = (signbit(d2) ? lo.z : hi.z) * rcp_approx(d2);
                        const float depth = fminf(t0, fminf(t1, t2));
                        if (dl[q] > 0.f) sum[k] += fabsf(dl[q] - depth);  // no pixel: dl = 0
                    }
                }
                // lanes with bit 16 (then 8) set carry the upper half of the poses on
#pragma unroll
                for (int o = 16, h = RC_GROUP / 2; h > 0; o >>= 1, h >>= 1)
#pragma unroll
                    for (int k = 0; k < h; ++k) {
                        const bool up = lane & o;
                        const float x = __shfl_xor_sync(0xffffffffu, up ? sum[k] : sum[k + h], o);
                        sum[k] = (up ? sum[k + h] : sum[k]) + x;
                    }
#pragma unroll
                for (int o = 16 / RC_GROUP; o > 0; o >>= 1) sum[0] += __shfl_xor_sync(0xffffffffu, sum[0], o);
                if ((lane & (32 / RC_GROUP - 1)) == 0) {
                    const int k = g + (lane >> 4 & 1) * 2 + (lane >> 3 & 1);
                    s_sum[k][w] = sum[0];
                    s_syn[k][w] = w_in;
                    s_both[k][w] = w_live;
                }
            }
        } else {
            for (int k = 0; k < cnt; ++k) {
                const float *P = sPf[k];
                float sum = 0.f;
                int syn = 0, both = 0;
                const float *E = s_exit[k];
                const bool in_box = E[0] < -1e-3f && E[4] > 1e-3f && E[1] < -1e-3f && E[5] > 1e-3f && E[2] < -1e-3f &&
                                    E[6] > 1e-3f;
#pragma unroll
                for (int q = 0; q < RC_PIX; ++q) {
                    if (!in[q]) continue;
                    float depth = 0.f;
                    if (in_box) {
                        const float d0 = fmaf(P[0], dc0[q], fmaf(P[1], dc1[q], P[2]));
                        const float d1 = fmaf(P[4], dc0[q], fmaf(P[5], dc1[q], P[6]));
                        const float d2 = fmaf(P[8], dc0[q], fmaf(P[9], dc1[q], P[10]));
                        const float t0 = (signbit(d0) ? E[0] : E[4]) * rcp_approx(d0);
                        const float t1 = (signbit(d1) ? E[1] : E[5]) * rcp_approx(d1);
                        const float t2 = (signbit(d2) ? E[2] : E[6]) * rcp_approx(d2);
                        depth = fminf(t0, fminf(t1, t2));
                    } else if (!ray_depth_slab(a, fr, P, a.pose_of(b, c0 + k), dc0[q], dc1[q], u[q], v[q], &depth, n64)) {
                        continue;
                    }
                    ++syn;
                    if (dl[q] > 0.f) {
                        ++both;
                        sum += fabsf(dl[q] - depth);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
                syn = __reduce_add_sync(0xffffffffu, syn);
                both = __reduce_add_sync(0xffffffffu, both);
                if (lane == 0) {
                    s_sum[k][w] = sum;
                    s_syn[k][w] = syn;
                    s_both[k][w] = both;
                }
            }
        }
        __syncthreads();
        if (threadIdx.x < cnt) {
            const int k = threadIdx.x;
            float ts = 0.f;
            int tsyn = 0, tb = 0;
            for (int ww = 0; ww < (int)(blockDim.x >> 5); ++ww) {
                ts += s_sum[k][ww];
                tsyn += s_syn[k][ww];
                tb += s_both[k][ww];
            }
            const size_t o = ((size_t)b * a.pose_cap + c0 + k) * a.n_tiles + blockIdx.x;
            a.part_sum[o] = (double)ts;
            a.part_cnt[2 * o] = tsyn;
            a.part_cnt[2 * o + 1] = tb;
        }
    }
    if (a.work) {
        if (threadIdx.x == 0)
            atomicAdd(&a.work[W_RAYS], (unsigned long long)n_poses *
                                           (unsigned long long)min(RC_TILE, npx - (int)(blockIdx.x * RC_TILE)));
        if (n64) atomicAdd(&a.work[W_RAY64], (unsigned long long)n64);
    }
}

// Eq. 7-8 per frame, then the frame's result record.  Eq. 7 for all chosen
// poses at once: tile partials summed by a fixed-shape block reduction (FP64
// sums, integer counts).  What bounds it is FP64 addition (one warp
// instruction in 64 cycles per sub-partition) and the latency of reading the
// partials, so the poses' sums are kept in flight together and meet at one
// barrier: 16 poses of 600 tiles 26 us, 51 with the poses one after another.
__global__ void __launch_bounds__(256) k_finalize(QueryState q, RParams p, int n_tiles, int ranked) {
    __shared__ double s_sum[16][8];
    __shared__ int s_syn[16][8], s_both[16][8];
    __shared__ float s_score[16];
    const int b = blockIdx.x;
    const Frame fr = q.frames[b];
    if (ranked && q.n_hyp[b] > 0) {
        const int nc = q.n_chosen[b], lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        for (int c0 = 0; c0 < nc; c0 += 4) {
            double sum[4] = {0.0, 0.0, 0.0, 0.0};
            int syn[4] = {0, 0, 0, 0}, both[4] = {0, 0, 0, 0};
            for (int t = threadIdx.x; t < n_tiles; t += blockDim.x)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const size_t o = ((size_t)b * 16 + min(c0 + k, nc - 1)) * n_tiles + t;
                    sum[k] += q.score_part[o];
                    const int2 cnt = ((const int2 *)q.score_cnt)[o];
                    syn[k] += cnt.x;
                    both[k] += cnt.y;
                }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int k = 0; k < 4; ++k) sum[k] += __shfl_down_sync(0xffffffffu, sum[k], o);
#pragma unroll
            for (int k = 0; k < 4; ++k) {  // at most 2^26 pixels: 32-bit counts
                syn[k] = __reduce_add_sync(0xffffffffu, syn[k]);
                both[k] = __reduce_add_sync(0xffffffffu, both[k]);
                if (lane == 0 && c0 + k < nc) {
                    s_sum[c0 + k][w] = sum[k];
                    s_syn[c0 + k][w] = syn[k];
                    s_both[c0 + k][w] = both[k];
                }
            }
        }
        __syncthreads();
        if ((int)threadIdx.x < nc) {
            const int c = threadIdx.x;
            double ts = 0.0;
            int tsyn = 0, tb = 0;
            for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
                ts += s_sum[c][k];
                tsyn += s_syn[c][k];
                tb += s_both[c][k];
            }
            const double frac = (double)tsyn / ((double)fr.W * (double)fr.H);
            // a pose whose ICP failed is discarded (Sec. 3.2.4)
            const bool kept = !p.icp || q.icp_ok[(size_t)b * 16 + c];
            const float sc = (kept && frac >= 0.1 && tb > 0) ? (float)(ts / (double)tb) : INFINITY;
            s_score[c] = sc;
            q.chosen_score[(size_t)b * 16 + c] = sc;
        }
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    DevResult *out = (DevResult *)q.result_blob + b;
    out->err = q.dev_err[b];
    out->n_hypotheses = q.n_hyp[b];
    out->n_chosen = q.n_hyp[b] > 0 ? q.n_chosen[b] : 0;
    out->n_pixels = q.n_pix[b];
    out->score = INFINITY;
    out->best = -1;
    out->icp_mask = 0;
    if (p.icp && q.n_hyp[b] > 0) {
        const int n_icp = ranked ? q.n_chosen[b] : 1;
        for (int c = 0; c < n_icp; ++c)
            if (q.icp_ok[(size_t)b * 16 + c]) out->icp_mask |= 1 << c;
    }
    if (q.n_hyp[b] == 0) {
        out->status = RL_NO_POSE;
        for (int k = 0; k < 12; ++k) out->pose[k] = (k % 5 == 0) ? 1.0 : 0.0;
        out->energy = INFINITY;
        out->energy_per_pixel = INFINITY;
        return;
    }
    out->status = RL_POSE_FOUND;
    const int NC = p.n_cull;
    int best = -1;
    float bs = INFINITY;
    if (ranked) {
        for (int c = 0; c < q.n_chosen[b]; ++c) {
            const float s = s_score[c];
            if (s < bs) {
                bs = s;
                best = c;
            }
        }
        if (best < 0) best = 0;
        out->score = bs;
        out->best = best;
        for (int k = 0; k < 12; ++k) out->pose[k] = q.chosen_pose[((size_t)b * 16 + best) * 12 + k];
        out->energy = q.chosen_energy[(size_t)b * 16 + best];
        out->energy_per_pixel = out->energy / (float)q.chosen_npix[b];
    } else {
        for (int c = 0; c < q.n_chosen[b]; ++c) q.chosen_score[(size_t)b * 16 + c] = INFINITY;
        for (int k = 0; k < 12; ++k) out->pose[k] = q.cur_pose[((size_t)b * NC) * 12 + k];
        out->energy = q.cur_energy[(size_t)b * NC];
        out->energy_per_pixel = out->energy / (float)q.n_pix[b];
    }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
rl_status launch_energy(const EnergyArgs &a0, int max_count, int n, cudaStream_t s, int max_threads) {
    EnergyArgs a = a0;
    int ht = 32;  // hypotheses per block: the smallest power of two covering them, capped
    while (ht < max_count && ht < max_threads) ht <<= 1;
    // A launch of one block per chunk and frame whose warps leave the GPU idle
    // gets threads beyond its hypotheses: lanes then share a hypothesis's mode
    // scan and the chunk is staged faster (the minimum is exact in any order).
    // Six 333x250 frames of 13 hypotheses: 15 us a round, 20 to 32 with the
    // hypotheses' own 64 threads.
    if (max_count <= ht)
        while (ht < 256 && (int64_t)((a.n_pix + a.chunk - 1) / a.chunk) * a.n_active * (ht / 32) * 2 <= 32 * (int64_t)a.sm_count)
            ht <<= 1;
    const size_t sm = (size_t)a.chunk * sizeof(float4) + (size_t)a.chunk * a.maxm * (2 * sizeof(float4) + sizeof(float)) +
                      (size_t)a.chunk * sizeof(int);
    dim3 grid((max_count + ht - 1) / ht, (a.n_pix + a.chunk - 1) / a.chunk, n);
    k_energy<<<grid, ht, sm, s>>>(a);
    RL_LAUNCH_CK();
    return RL_OK;
}

size_t energy_smem(int chunk, int maxm) {
    return (size_t)chunk * sizeof(float4) + (size_t)chunk * maxm * (2 * sizeof(float4) + sizeof(float)) +
           (size_t)chunk * sizeof(int);
}

rl_status launch_select(const SelectArgs &a, int n, cudaStream_t s) {
    const size_t sm = (size_t)a.p.n_hyp * (sizeof(float) + sizeof(int)) +
                      (size_t)a.p.n_cull * (12 * sizeof(double) + sizeof(float) + sizeof(int)) + 64;
    k_select<<<n, 1024, sm, s>>>(a);
    RL_LAUNCH_CK();
    return RL_OK;
}

bool lm_uses_cluster(const RParams &p) {
    return p.n_cull <= 64 && lm_cluster_smem(p.mpad, p.use_cov) <= kLmClusterSmemMax;
}

// The cluster kernel, or (rows too long for its staged tiles) the spread
// kernel; n_cull <= 64 (checked when the relocaliser is created).
rl_status launch_lm(const LmArgs &a, int n, cudaStream_t s) {
    if (lm_uses_cluster(a.p)) return launch_lm_cluster(a, n, s);
    const int fit = 2 * a.sm_count / LM3_BPQ;  // parts of one block each that fit two blocks per SM
    if (8 * a.n_active <= fit) return launch_lm_spread<8>(a, n, s);
    if (4 * a.n_active <= fit) return launch_lm_spread<4>(a, n, s);
    if (2 * a.n_active <= fit) return launch_lm_spread<2>(a, n, s);
    return launch_lm_spread<1>(a, n, s);
}

// Kernel attributes set once, outside any stream capture.
rl_status prepare_kernels() {
    static bool done = false;
    static std::mutex mu;
    std::lock_guard<std::mutex> g(mu);
    if (done) return RL_OK;
    RL_TRY(prepare_lm_cluster());
    RL_TRY(prepare_hypgen());
    done = true;
    return RL_OK;
}

rl_status launch_raycast(const RaycastArgs &a, int n, int max_hw, cudaStream_t s) {
    dim3 grid(a.n_tiles, n);
    k_raycast_score<<<grid, 256, 0, s>>>(a);
    RL_LAUNCH_CK();
    return RL_OK;
}

rl_status launch_finalize(const QueryState &q, const RParams &p, int n_tiles, int ranked, int n,
                          cudaStream_t s) {
    k_finalize<<<n, 256, 0, s>>>(q, p, n_tiles, ranked);
    RL_LAUNCH_CK();
    return RL_OK;
}

}  // namespace rl

namespace rl {
// Standalone Eq. 6-7 scorer: poses [n][12] against one live depth frame.  A
// warp per pose sums its tile partials in FP64 (one thread walking all tiles
// took 83 us for 128 poses at 640x480, the lanes 8 us).
__global__ void __launch_bounds__(128) k_scores_final(const double *__restrict__ part_sum,
                                                      const int32_t *__restrict__ part_cnt, int n_tiles, int n,
                                                      double npx, float *__restrict__ scores,
                                                      float *__restrict__ valid_frac) {
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= n) return;
    double sum = 0.0;
    int syn = 0, both = 0;
    for (int t = lane; t < n_tiles; t += 32) {
        const size_t o = (size_t)c * n_tiles + t;
        sum += part_sum[o];
        const int2 cnt = ((const int2 *)part_cnt)[o];
        syn += cnt.x;
        both += cnt.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    syn = __reduce_add_sync(0xffffffffu, syn);
    both = __reduce_add_sync(0xffffffffu, both);
    if (lane != 0) return;
    const double frac = (double)syn / npx;
    valid_frac[c] = (float)frac;
    scores[c] = (frac >= 0.1 && both > 0) ? (float)(sum / (double)both) : INFINITY;
}

rl_status launch_score_poses(const RaycastArgs &a, int n_poses, int npx, float *scores,
                             float *valid_frac, cudaStream_t s) {
    dim3 grid(a.n_tiles, 1);
    k_raycast_score<<<grid, 256, 0, s>>>(a);
    RL_LAUNCH_CK();
    k_scores_final<<<(n_poses + 3) / 4, 128, 0, s>>>(a.part_sum, a.part_cnt, a.n_tiles, n_poses,
                                                      (double)npx, scores, valid_frac);
    RL_LAUNCH_CK();
    return RL_OK;
}
}  // namespace rl
