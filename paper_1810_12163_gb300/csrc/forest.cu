// Random forest factory (Sec. 4.5), split features and forest walk
// (Eq. 1-3), and deterministic online reservoir adaptation (Sec. 3.2.2).
//
// Compiled with --fmad=false: the FP32 feature arithmetic and the FP64
// back-projection are plain IEEE operations in a fixed order, so leaves and
// reservoir contents are exactly reproducible.
#include <cooperative_groups.h>

#include <algorithm>

#include "internal.h"
#include "relocgb_dev.cuh"

namespace rl {

__device__ __forceinline__ float unit24(uint32_t u) {
    return __fmul_rn((float)(u >> 8), 1.0f / 16777216.0f);
}

// One thread per branch node.  Two Philox blocks per node: (type draw, dx,
// dy, channel) and (tau).
__global__ void k_forest_random(float4 *nodes, int n_trees, int n_branch, float p_depth,
                                float dlo, float dhi, float tdlo, float tdhi, float trlo,
                                float trhi, int tau_zero, uint32_t k0, uint32_t k1) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_trees * n_branch) return;
    const int t = i / n_branch, n = i % n_branch;
    const uint4 r0 = philox(make_uint4(t, TAG_FOREST << 16, n, 0), k0, k1);
    const uint4 r1 = philox(make_uint4(t, TAG_FOREST << 16, n, 1), k0, k1);
    const bool is_depth = (double)r0.x < (double)p_depth * 4294967296.0;
    const float span = __fsub_rn(dhi, dlo);
    float4 nd;
    nd.x = __fadd_rn(dlo, __fmul_rn(span, unit24(r0.y)));
    nd.y = __fadd_rn(dlo, __fmul_rn(span, unit24(r0.z)));
    float tau = 0.0f;
    if (!tau_zero) {
        const float lo = is_depth ? tdlo : trlo, hi = is_depth ? tdhi : trhi;
        tau = __fadd_rn(lo, __fmul_rn(__fsub_rn(hi, lo), unit24(r1.x)));
    }
    nd.z = tau;
    const uint32_t meta = is_depth ? 0u : (1u | (draw_below(r0.w, 3) << 8));
    nd.w = __uint_as_float(meta);
    nodes[i] = nd;
}

rl_status launch_forest_random(rl_forest *f, cudaStream_t s) {
    const rl_forest_params &p = f->p;
    const int n = p.n_trees * f->n_branch;
    k_forest_random<<<(n + 255) / 256, 256, 0, s>>>(
        f->nodes, p.n_trees, f->n_branch, p.p_depth, p.delta_lo, p.delta_hi, p.tau_depth_lo,
        p.tau_depth_hi, p.tau_rgb_lo, p.tau_rgb_hi, p.tau_zero, (uint32_t)f->seed,
        (uint32_t)(f->seed >> 32));
    RL_LAUNCH_CK();
    return RL_OK;
}

// ---------------------------------------------------------------------------
// Eq. 1-3.  Probe q = p + delta * (fx / 585) / D(p), rounded to the nearest
// pixel and clamped to the image; a Depth split compares D(p) - D(q), a
// DA-RGB split C(p,c) - C(q,c), against tau; true goes right (2n+2).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int probe_coord(int p, float off, int extent) {
    const float v = __fadd_rn(__fadd_rn((float)p, off), 0.5f);
    // floor to an integer (saturating beyond the int range, 0 for NaN), then
    // clamp: the same as clamping floor(v) in FP32 and converting
    return min(max(__float2int_rd(v), 0), extent - 1);
}

__device__ __forceinline__ int walk_tree(const float4 *__restrict__ nodes, int depth,
                                         const float *__restrict__ D, const uint8_t *__restrict__ C,
                                         int W, int H, float s, int x, int y, float d, float inv) {
    int n = 0;
    const int p = y * W + x;
    for (int level = 0; level < depth; ++level) {
        const float4 nd = __ldg(&nodes[n]);
        const uint32_t meta = __float_as_uint(nd.w);
        const float ox = __fmul_rn(__fmul_rn(nd.x, s), inv);
        const float oy = __fmul_rn(__fmul_rn(nd.y, s), inv);
        const int qx = probe_coord(x, ox, W);
        const int qy = probe_coord(y, oy, H);
        const int q = qy * W + qx;
        float f;
        if ((meta & 255u) == 0u) {
            const float dq = __ldg(&D[q]);
            f = __fsub_rn(d, dq > 0.0f ? dq : 0.0f);
        } else {
            const int c = (int)(meta >> 8);
            f = __fsub_rn((float)__ldg(&C[p * 3 + c]), (float)__ldg(&C[q * 3 + c]));
        }
        n = (f >= nd.z) ? 2 * n + 2 : 2 * n + 1;
    }
    return n - ((1 << depth) - 1);
}

// A call's node (k_scale_nodes): offsets times fx / 585, and for the split
// either kSplitDepth or the selector of a byte permute that makes the float
// 2^23 + c of the channel's colour byte c; its low 4 bits are the channel.
constexpr uint32_t kSplitDepth = 0x80000000u;
constexpr uint32_t kSplitByte = 0x7540u;  // bytes c, 0x00, 0x00, 0x4B of (colours, 0x4B000000)

// All T trees of one pixel walked level by level, interleaved: T
// independent chains of dependent node and probe loads in flight at once.
// PRE: the nodes are a call's.
template <int T, bool PRE>
__device__ __forceinline__ void walk_trees(const float4 *__restrict__ nodes, int n_branch, int depth,
                                           const float *__restrict__ D, const uint8_t *__restrict__ C,
                                           int W, int H, float s, int x, int y, float d, float inv,
                                           int leaf[T]) {
    int n[T];
#pragma unroll
    for (int t = 0; t < T; ++t) n[t] = 0;
    const int p = y * W + x;
    for (int level = 0; level < depth; ++level) {
        float4 nd[T];
#pragma unroll
        for (int t = 0; t < T; ++t) nd[t] = __ldg(&nodes[(size_t)t * n_branch + n[t]]);
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const uint32_t meta = __float_as_uint(nd[t].w);
            const float ox = __fmul_rn(PRE ? nd[t].x : __fmul_rn(nd[t].x, s), inv);
            const float oy = __fmul_rn(PRE ? nd[t].y : __fmul_rn(nd[t].y, s), inv);
            const int q = probe_coord(y, oy, H) * W + probe_coord(x, ox, W);
            float f;
            if (PRE ? meta == kSplitDepth : (meta & 255u) == 0u) {
                const float dq = __ldg(&D[q]);
                f = __fsub_rn(d, dq > 0.0f ? dq : 0.0f);
            } else {
                const int c = (int)(PRE ? meta & 15u : meta >> 8);
                f = __fsub_rn((float)__ldg(&C[p * 3 + c]), (float)__ldg(&C[q * 3 + c]));
            }
            n[t] = (f >= nd[t].z) ? 2 * n[t] + 2 : 2 * n[t] + 1;
        }
    }
#pragma unroll
    for (int t = 0; t < T; ++t) leaf[t] = n[t] - ((1 << depth) - 1);
}

template <int T, bool PRE>
__device__ __forceinline__ int walk_and_store(const float4 *nodes, int n_branch, int depth, const Frame &fr,
                                              float s, int x, int y, float d, float inv, uint16_t *o,
                                              int hw_max, const uint8_t *nmodes, int lpt, int k_top,
                                              bool count, uint4 *rec) {
    int leaf[kRecTrees], cnt[kRecTrees];
    walk_trees<T, PRE>(nodes, n_branch, depth, fr.depth, fr.rgb, fr.W, fr.H, s, x, y, d, inv, leaf);
    int total = 0;
#pragma unroll
    for (int t = 0; t < T; ++t) {
        if (o) o[(size_t)t * hw_max] = (uint16_t)leaf[t];
        cnt[t] = count ? min((int)__ldg(&nmodes[t * lpt + leaf[t]]), k_top) : 0;
        total += cnt[t];
    }
    if (rec) *rec = make_rec(leaf, cnt, T);
    return total;
}

// out: uint16 [frame][tree][hw_max] (null: not written); one thread per
// pixel walks every tree.
// When `mcount` is given it also receives |M(u)| = sum over the trees of
// min(modes of the reached leaf, k_top) per pixel (0 without depth); the
// pixel records `prec` (at most kRecTrees trees) hold the per-tree counts.
// nodes_s: the call's nodes for focal length fx_s, taken for the frames of
// that focal length, or null.
__global__ void k_leaves(const float4 *__restrict__ nodes, int n_branch, int depth, int n_trees,
                         const Frame *__restrict__ frames, int hw_max, uint16_t *__restrict__ out,
                         const uint8_t *__restrict__ nmodes, int leaves_per_tree, int k_top,
                         uint16_t *__restrict__ mcount, uint4 *__restrict__ prec,
                         const float4 *__restrict__ nodes_s, float fx_s) {
    const Frame fr = frames[blockIdx.y];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= fr.W * fr.H) return;
    const int x = p % fr.W, y = p / fr.W;
    const float d = __ldg(&fr.depth[p]);
    uint16_t *o = out ? out + (size_t)blockIdx.y * n_trees * hw_max + p : nullptr;  // null: no leaf map
    uint4 *rec = prec ? prec + (size_t)blockIdx.y * hw_max + p : nullptr;
    if (!(d > 0.0f)) {
        if (o)
            for (int t = 0; t < n_trees; ++t) o[(size_t)t * hw_max] = 0xFFFF;
        if (mcount) mcount[(size_t)blockIdx.y * hw_max + p] = 0;
        if (rec) *rec = make_uint4(0, 0, 0, 0);
        return;
    }
    const float s = __fdiv_rn(fr.fx, 585.0f);
    const float inv = __frcp_rn(d);
    int total = 0;
    const bool cnt = mcount != nullptr || prec != nullptr;  // per-tree counts wanted
    const bool pre = nodes_s != nullptr && fr.fx == fx_s;   // the same for the whole block (one frame)
#define RL_WALK(T)                                                                                          \
    total = pre ? walk_and_store<T, true>(nodes_s, n_branch, depth, fr, s, x, y, d, inv, o, hw_max, nmodes, \
                                          leaves_per_tree, k_top, cnt, rec)                                  \
                : walk_and_store<T, false>(nodes, n_branch, depth, fr, s, x, y, d, inv, o, hw_max, nmodes,  \
                                           leaves_per_tree, k_top, cnt, rec)
    switch (n_trees) {
    case 1: RL_WALK(1); break;
    case 2: RL_WALK(2); break;
    case 3: RL_WALK(3); break;
    case 4: RL_WALK(4); break;
    case 5: RL_WALK(5); break;
#undef RL_WALK
    default:
        for (int t = 0; t < n_trees; ++t) {
            const int leaf = walk_tree(nodes + (size_t)t * n_branch, depth, fr.depth, fr.rgb, fr.W, fr.H,
                                       s, x, y, d, inv);
            if (o) o[(size_t)t * hw_max] = (uint16_t)leaf;
            if (cnt) total += min((int)__ldg(&nmodes[t * leaves_per_tree + leaf]), k_top);
        }
    }
    if (mcount) mcount[(size_t)blockIdx.y * hw_max + p] = (uint16_t)total;
}

rl_status launch_leaves(const rl_forest *f, const Frame *frames_dev, int n_frames, int n_trees,
                        int hw_max, uint16_t *out, int max_w, int max_h, cudaStream_t s,
                        int k_top, uint16_t *mcount, uint4 *prec, int threads, const float4 *nodes_s,
                        float fx_s) {
    const int npx = max_w * max_h;
    dim3 grid((npx + threads - 1) / threads, n_frames);
    k_leaves<<<grid, threads, 0, s>>>(f->nodes, f->n_branch, f->p.depth, n_trees, frames_dev, hw_max, out,
                                  f->nmodes, f->leaves_per_tree, k_top, mcount,
                                  n_trees <= kRecTrees ? prec : nullptr, nodes_s, fx_s);
    RL_LAUNCH_CK();
    return RL_OK;
}

// ---------------------------------------------------------------------------
// The walk of a relocalisation call (at most kRecTrees trees, pixel records
// out).  It is bound by issue: 75 node tests per pixel of exact FP32 feature
// arithmetic whose gathers mostly hit L1.  Three things keep a test short:
//  - frames are packed first, 8 bytes per pixel (depth, 0 where invalid; the
//    three colours), so a probe is one gather whatever the split tests;
//  - both kinds of split are evaluated without a branch (below the first
//    levels a warp's lanes differ): a colour byte c becomes the float 2^23 +
//    c by one byte permute, and the difference of two such floats is exactly
//    the difference of the colours;
//  - the call's nodes carry the offsets times fx / 585 and the permute's
//    selector, and a coordinate is clamped by one min-with-relu.
// It needs 8 bytes per pixel that nothing else uses yet (run_relocalise);
// k_leaves walks the frames as they are where there is no such place.
// That is 33 instructions a test instead of 44.  Measured on 8 frames of
// 640x480, 5 trees of depth 15: 208 us + 11 us of packing (was 267; 75% issue,
// the gathers' latency next), one frame 38 + 4 us (51).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float4 pack_node(float4 v, float s) {
    const uint32_t meta = __float_as_uint(v.w);
    const uint32_t sel = (meta & 255u) == 0u ? kSplitDepth : kSplitByte | (meta >> 8);
    return make_float4(__fmul_rn(v.x, s), __fmul_rn(v.y, s), v.z, __uint_as_float(sel));
}

// frame b's pixels at out + b * hw_max
__global__ void __launch_bounds__(256) k_pack_frames(const Frame *__restrict__ frames, uint2 *__restrict__ out,
                                                     int hw_max) {
    const Frame fr = frames[blockIdx.y];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= fr.W * fr.H) return;
    const float d = fr.depth[p];
    const uint8_t *c = fr.rgb + (size_t)p * 3;
    out[(size_t)blockIdx.y * hw_max + p] = make_uint2(__float_as_uint(d > 0.0f ? d : 0.0f),
                                              (uint32_t)c[0] | ((uint32_t)c[1] << 8) | ((uint32_t)c[2] << 16));
}

// nodes: packed for focal length fx_s when PRE, else the forest's
template <int T, bool PRE>
__device__ __forceinline__ uint4 walk_packed(const float4 *__restrict__ nodes, int n_branch, int depth,
                                             const uint2 *__restrict__ px, int W, int H, float s, int x, int y,
                                             uint2 own, float inv, const uint8_t *__restrict__ nmodes, int lpt,
                                             int k_top) {
    int n[T];
#pragma unroll
    for (int t = 0; t < T; ++t) n[t] = 0;
    const float d = __uint_as_float(own.x);
    const float fx = (float)x, fy = (float)y;
    for (int level = 0; level < depth; ++level) {
        float4 nd[T];
#pragma unroll
        for (int t = 0; t < T; ++t) nd[t] = __ldg(&nodes[(size_t)t * n_branch + n[t]]);
#pragma unroll
        for (int t = 0; t < T; ++t) {
            if (!PRE) nd[t] = pack_node(nd[t], s);
            const float vx = __fadd_rn(__fadd_rn(fx, __fmul_rn(nd[t].x, inv)), 0.5f);
            const float vy = __fadd_rn(__fadd_rn(fy, __fmul_rn(nd[t].y, inv)), 0.5f);
            const int qx = __vimin_s32_relu(__float2int_rd(vx), W - 1), qy = __vimin_s32_relu(__float2int_rd(vy), H - 1);
            const uint2 w = __ldg(&px[qy * W + qx]);
            const uint32_t sel = __float_as_uint(nd[t].w);
            const float fd = __fsub_rn(d, __uint_as_float(w.x));
            const float fc = __fsub_rn(__uint_as_float(__byte_perm(own.y, 0x4B000000u, sel)),
                                       __uint_as_float(__byte_perm(w.y, 0x4B000000u, sel)));
            n[t] = 2 * n[t] + (((int)sel < 0 ? fd : fc) >= nd[t].z ? 2 : 1);
        }
    }
    int leaf[kRecTrees], cnt[kRecTrees];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        leaf[t] = n[t] - ((1 << depth) - 1);
        cnt[t] = min((int)__ldg(&nmodes[t * lpt + leaf[t]]), k_top);
    }
    return make_rec(leaf, cnt, T);
}

template <int T>
__global__ void k_leaves_packed(const float4 *__restrict__ nodes, const float4 *__restrict__ nodes_s, float fx_s,
                                int n_branch, int depth, const Frame *__restrict__ frames, int hw_max,
                                const uint2 *__restrict__ packed, const uint8_t *__restrict__ nmodes,
                                int leaves_per_tree, int k_top, uint4 *__restrict__ prec) {
    const Frame fr = frames[blockIdx.y];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= fr.W * fr.H) return;
    const uint2 *px = packed + (size_t)blockIdx.y * hw_max;
    const uint2 own = px[p];
    const float d = __uint_as_float(own.x);
    uint4 rec = make_uint4(0, 0, 0, 0);
    if (d > 0.0f) {
        const int x = p % fr.W, y = p / fr.W;
        const float s = __fdiv_rn(fr.fx, 585.0f);
        const float inv = __frcp_rn(d);
        // the same for the whole block (one frame)
        rec = fr.fx == fx_s ? walk_packed<T, true>(nodes_s, n_branch, depth, px, fr.W, fr.H, s, x, y, own, inv, nmodes,
                                                   leaves_per_tree, k_top)
                            : walk_packed<T, false>(nodes, n_branch, depth, px, fr.W, fr.H, s, x, y, own, inv, nmodes,
                                                    leaves_per_tree, k_top);
    }
    prec[(size_t)blockIdx.y * hw_max + p] = rec;
}

rl_status launch_leaves_packed(const rl_forest *f, const Frame *frames_dev, int n_frames, int n_trees, int hw_max,
                               cudaStream_t s, int k_top, uint4 *prec, int threads, const float4 *nodes_s, float fx_s,
                               uint2 *packed) {
    k_pack_frames<<<dim3((hw_max + 255) / 256, n_frames), 256, 0, s>>>(frames_dev, packed, hw_max);
    RL_LAUNCH_CK();
    const dim3 grid((hw_max + threads - 1) / threads, n_frames);
#define RL_WALK(T)                                                                                                 \
    k_leaves_packed<T><<<grid, threads, 0, s>>>(f->nodes, nodes_s, fx_s, f->n_branch, f->p.depth, frames_dev, hw_max, \
                                                packed, f->nmodes, f->leaves_per_tree, k_top, prec)
    switch (n_trees) {
    case 1: RL_WALK(1); break;
    case 2: RL_WALK(2); break;
    case 3: RL_WALK(3); break;
    case 4: RL_WALK(4); break;
    default: RL_WALK(5); break;
    }
#undef RL_WALK
    RL_LAUNCH_CK();
    return RL_OK;
}

// A call's split nodes: offsets multiplied by s = fx / 585 (Eq. 1-3's
// depth-normalised probe offset), rounded as the walk rounds its own first
// product, and the split in the walk's form.
__global__ void k_scale_nodes(const float4 *__restrict__ nodes, float4 *__restrict__ out, int count, float fx) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) out[i] = pack_node(nodes[i], __fdiv_rn(fx, 585.0f));
}

rl_status launch_scale_nodes(const rl_forest *f, int n_trees, float4 *out, float fx, cudaStream_t s) {
    const int count = n_trees * f->n_branch;
    k_scale_nodes<<<(count + 255) / 256, 256, 0, s>>>(f->nodes, out, count, fx);
    RL_LAUNCH_CK();
    return RL_OK;
}

// ---------------------------------------------------------------------------
// Reservoir adaptation (Sec. 3.2.2), deterministic Algorithm R.
//
// For one frame: (1) every grid pixel with depth is back-projected, moved to
// world space and walked down every tree, and its leaves count it.  (2) Every
// leaf gets a segment of the frame's example list, in leaf order, and its
// reservoir's count goes up by the segment's length.  (3) The examples are
// scattered into their leaf's segment (in any order).  (4) An example's rank
// among the frame's examples of its leaf, in pixel order, is the number of
// smaller pixels in its segment; it gives the count c = count_before_frame +
// rank and, with it, Algorithm R's slot, a pure function of (leaf, c).  (5)
// An example writes its slot unless a later example of the same leaf in this
// frame draws the same slot.
//
// Scratch is two words per example (list entry; leaf and slot of 16 bits) and
// the points.  A segment needs no record of its own: step 3 advances a leaf's
// count from where its segment starts to where it ends, and it starts where
// the leaf before ends.
//
// Threads of steps 4 and 5 follow the list, so that the lanes of a warp
// mostly look at one segment.  Segments shorter than EX_WIDE are staged in
// shared memory and read by broadcast, each example against all the others.
// A longer one (a thousand or two in the fullest leaf of a room) gets a table
// in every block that holds a part of it: a bitmap of its pixels, whose
// running count is the rank, and the last pixel of each slot.
// Measured on GB300 (640x480, 19,200 grid pixels, 5 trees of depth 15): 33 us
// a frame (clearing 1.5, walk 11, segments 5, scatter 2.5, slots 7, insert
// 6.5), a call 47 us; of depth 11 a call is 43 us, of depth 6 43 (59 with an
// atomic per example, whose leaves are then full).  With a record per segment
// and words of their own for arrival numbers and slots, 4 bytes more per
// example and 8 per leaf, the calls took 48, 47 and 59 us.  Every entry
// against every other in long segments too: 18 us slots, 27 us insert.  A
// thread per pixel walking all trees, ranks from all pairs of pixels and the
// slot of every later example drawn again: 620 us.
// ---------------------------------------------------------------------------
constexpr int EX_THREADS = 128, EX_TILE = 1024;
constexpr int EX_WIDE = 256;      // entries from which a segment gets a table
constexpr int EX_TABLE = 4096;    // its words: 131,072 pixels at a time, or the largest capacity
constexpr uint16_t kNoLeaf = 0xFFFFu, kNoSlot = 0xFFFFu;  // a tree has at most 2^15, capacities are at most 4096
constexpr int EX_SCAN_THREADS = 1024, EX_SCAN_EACH = 4;  // eight blocks: 2^15 leaves, the most a tree has

struct Pose12 {
    double m[12];
};

__global__ void k_adapt_examples(const float4 *__restrict__ nodes, int n_branch, int depth,
                                 int leaves_per_tree, const float *__restrict__ D,
                                 const uint8_t *__restrict__ C, int W, int H, float fx, float fy,
                                 float cx, float cy, Pose12 T, int gw, int gh, int step, int origin,
                                 uint16_t *__restrict__ ex_leaf, float4 *__restrict__ ex_pt,
                                 uint32_t *__restrict__ frame_cnt) {
    const int P = gw * gh;
    const int g = blockIdx.x * blockDim.x + threadIdx.x, t = blockIdx.y;  // a thread per (grid pixel, tree)
    const int x = origin + (g % gw) * step, y = origin + (g / gw) * step;
    const int p = y * W + x;
    const float d = g < P ? D[p] : 0.0f;
    const size_t e = (size_t)t * P + g;
    const unsigned live = __ballot_sync(0xffffffffu, d > 0.0f);
    if (!(d > 0.0f)) {
        if (g < P) ex_leaf[e] = kNoLeaf;
        return;
    }
    if (t == 0) {
        const float xc = __fdiv_rn(__fmul_rn(__fsub_rn((float)x, cx), d), fx);
        const float yc = __fdiv_rn(__fmul_rn(__fsub_rn((float)y, cy), d), fy);
        const float zc = d;
        float w[3];
        for (int r = 0; r < 3; ++r) {
            const double a = __dmul_rn(T.m[4 * r + 0], (double)xc);
            const double b = __dmul_rn(T.m[4 * r + 1], (double)yc);
            const double c = __dmul_rn(T.m[4 * r + 2], (double)zc);
            w[r] = (float)__dadd_rn(__dadd_rn(__dadd_rn(a, b), c), T.m[4 * r + 3]);
        }
        const uint32_t rgb = (uint32_t)C[3 * p] | ((uint32_t)C[3 * p + 1] << 8) | ((uint32_t)C[3 * p + 2] << 16);
        ex_pt[g] = make_float4(w[0], w[1], w[2], __uint_as_float(rgb));
    }
    const float s = __fdiv_rn(fx, 585.0f);
    const float inv = __frcp_rn(d);
    const int leaf = walk_tree(nodes + (size_t)t * n_branch, depth, D, C, W, H, s, x, y, d, inv);
    ex_leaf[e] = (uint16_t)leaf;
    // one atomic for a warp's examples of a leaf: neighbours often share it,
    // and those of a full leaf would queue at its count
    const unsigned same = __match_any_sync(live, leaf);
    if ((threadIdx.x & 31) == __ffs(same) - 1)
        atomicAdd(&frame_cnt[t * leaves_per_tree + leaf], (uint32_t)__popc(same));
}

// Segments: each count of a tree's leaves becomes where the leaf's segment
// starts, the sum of the counts before it (tree t's segments lie in [t P, (t +
// 1) P)), and is added to the leaf's reservoir count.  A cluster of blocks per
// tree (one block up to 4,096 leaves), so that any tree takes one step of it.
__global__ void __launch_bounds__(EX_SCAN_THREADS)
    k_adapt_segments(uint32_t *__restrict__ frame_cnt, uint32_t *__restrict__ res_count, int leaves_per_tree, int P) {
    __shared__ uint32_t sums[32], total;
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, rank = blockIdx.x, t = blockIdx.y;
    const int per = EX_SCAN_EACH * blockDim.x;  // a block's leaves
    const int l0 = rank * per + EX_SCAN_EACH * tid, end = leaves_per_tree;
    uint32_t *cnt = frame_cnt + (size_t)t * leaves_per_tree, *res = res_count + (size_t)t * leaves_per_tree;
    uint32_t c[EX_SCAN_EACH], before[EX_SCAN_EACH], mine = 0;
#pragma unroll
    for (int k = 0; k < EX_SCAN_EACH; ++k) {
        c[k] = l0 + k < end ? cnt[l0 + k] : 0;
        before[k] = l0 + k < end ? res[l0 + k] : 0;
    }
#pragma unroll
    for (int k = 0; k < EX_SCAN_EACH; ++k) mine += c[k];
    auto sum_to = [&](uint32_t v) {  // over the warp's lanes up to this one
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += x;
        }
        return v;
    };
    const uint32_t upto = sum_to(mine);
    if (lane == 31) sums[w] = upto;
    __syncthreads();
    if (w == 0) {
        const uint32_t v = lane < (int)blockDim.x / 32 ? sums[lane] : 0, all = sum_to(v);
        sums[lane] = all - v;
        if (lane == 31) total = all;
    }
    __syncthreads();
    if (gridDim.x > 1) cluster.sync();
    uint32_t at = (uint32_t)t * (uint32_t)P + sums[w] + upto - mine;
    // the blocks before, a lane each (at most eight blocks)
    at += __reduce_add_sync(0xffffffffu, lane < rank ? *cluster.map_shared_rank(&total, lane) : 0u);
#pragma unroll
    for (int k = 0; k < EX_SCAN_EACH; ++k)
        if (l0 + k < end) {
            cnt[l0 + k] = at;
            if (c[k]) res[l0 + k] = before[k] + c[k];
            at += c[k];
        }
    if (gridDim.x > 1) cluster.sync();  // no block leaves while another may still read its sum
}

__global__ void k_adapt_scatter(const uint16_t *__restrict__ ex_leaf, int P, int leaves_per_tree,
                                uint32_t *__restrict__ frame_cnt, uint32_t *__restrict__ list) {
    const int g = blockIdx.x * blockDim.x + threadIdx.x, t = blockIdx.y, lane = threadIdx.x & 31;
    const uint32_t leaf = g < P ? ex_leaf[(size_t)t * P + g] : kNoLeaf;
    const unsigned same = __match_any_sync(0xffffffffu, leaf);
    const int first = __ffs(same) - 1;
    uint32_t at = 0;
    if (lane == first && leaf != kNoLeaf) at = atomicAdd(&frame_cnt[t * leaves_per_tree + leaf], (uint32_t)__popc(same));
    at = __shfl_sync(0xffffffffu, at, first);
    if (leaf != kNoLeaf) list[at + __popc(same & ((1u << lane) - 1u))] = (uint32_t)g;
}

// What a step reads of the list once it is filled.
struct ExList {
    const uint32_t *entry;  // grid pixels, tree t's from t P
    const uint32_t *ends;   // [L] end of the leaf's segment
    int P, leaves_per_tree;
    // entries [t P, end(t)) are in use
    __device__ uint32_t end(int t) const { return ends[(t + 1) * leaves_per_tree - 1]; }
    // (first entry, length) of leaf `leaf` of tree t
    __device__ uint2 segment(int t, uint32_t leaf) const {
        const uint32_t l = (uint32_t)(t * leaves_per_tree) + leaf;
        const uint32_t first = leaf ? ends[l - 1] : (uint32_t)t * (uint32_t)P;
        return make_uint2(first, ends[l] - first);
    }
};

__device__ __forceinline__ int64_t reservoir_slot(uint32_t L, uint32_t c, int kappa, uint32_t k0,
                                                  uint32_t k1) {
    if (c < (uint32_t)kappa) return c;
    const uint4 r = philox(make_uint4(L, TAG_RESERVOIR << 16, c, 0), k0, k1);
    const uint64_t j = ((uint64_t)r.x * ((uint64_t)c + 1)) >> 32;
    return j < (uint64_t)kappa ? (int64_t)j : -1;
}

// Runs f(first, last) on every thread of a block for the part of its segment
// [sg.x, sg.x + sg.y) in each tile of the block's segments (load(q0, n) stages
// entries q0 .. q0 + n in shared memory); threads without a segment have
// sg.y = 0.  Every thread of the block calls it.
template <class Load, class F>
__device__ __forceinline__ void segment_tiles(uint2 sg, Load load, F f) {
    __shared__ uint32_t lo, hi;
    if (threadIdx.x == 0) {
        lo = 0xFFFFFFFFu;
        hi = 0;
    }
    __syncthreads();
    const uint32_t end = sg.x + sg.y;
    if (sg.y) {
        atomicMin(&lo, sg.x);
        atomicMax(&hi, end);
    }
    __syncthreads();
    const uint32_t q1 = hi;
    for (uint32_t q0 = lo; q0 < q1; q0 += EX_TILE) {
        const uint32_t n = min((uint32_t)EX_TILE, q1 - q0);
        load(q0, n);
        __syncthreads();
        const uint32_t first = max(q0, sg.x), last = min(q0 + n, end);
        if (first < last) f(first - q0, last - q0);
        __syncthreads();
    }
}

// Runs f(segment) for the segments of EX_WIDE entries or more that the block
// holds a part of: sg is the segment of the thread's entry, live >= 1 the
// block's entries.  Being longer than a block, such a segment holds the
// block's first entry or its last.
template <class F>
__device__ __forceinline__ void wide_segments(uint2 sg, uint32_t live, F f) {
    static_assert(EX_WIDE >= EX_THREADS, "at most two wide segments in a block");
    __shared__ uint2 ends[2];
    if (threadIdx.x == 0) ends[0] = sg;
    if (threadIdx.x == live - 1) ends[1] = sg;
    __syncthreads();
    const uint2 a = ends[0], b = ends[1];
    if (a.y >= EX_WIDE) f(a);
    if (b.y >= EX_WIDE && b.x != a.x) f(b);
}

// slot[r]: the slot of entry r of the list, or kNoSlot.
__global__ void __launch_bounds__(EX_THREADS) k_adapt_slots(const uint16_t *__restrict__ ex_leaf, ExList list,
                                                            const uint32_t *__restrict__ res_count, int kappa,
                                                            uint32_t k0, uint32_t k1, uint16_t *__restrict__ slot) {
    __shared__ uint32_t s_g[EX_TILE], table[EX_TABLE], chunk[EX_THREADS], sum[EX_THREADS / 32];
    const int P = list.P, t = blockIdx.y;
    const uint32_t r0 = (uint32_t)t * P + blockIdx.x * EX_THREADS, r = r0 + threadIdx.x, end = list.end(t);
    if (r0 >= end) return;
    const bool on = r < end;
    const uint32_t g = on ? list.entry[r] : 0;
    const uint32_t leaf = on ? ex_leaf[(size_t)t * P + g] : 0;
    const uint2 sg = on ? list.segment(t, leaf) : make_uint2(0, 0);
    uint32_t rank = 0;
    wide_segments(sg, min(end - r0, (uint32_t)EX_THREADS), [&](uint2 e) {
        for (uint32_t w0 = 0; w0 < (uint32_t)P; w0 += EX_TABLE * 32) {  // the set bits below g
            const uint32_t words = min((uint32_t)EX_TABLE, ((uint32_t)P - w0 + 31) / 32);
            for (uint32_t i = threadIdx.x; i < words; i += EX_THREADS) table[i] = 0;
            __syncthreads();
            for (uint32_t q = threadIdx.x; q < e.y; q += EX_THREADS) {
                const uint32_t d = list.entry[e.x + q] - w0;
                if (d < words * 32) atomicOr(&table[d >> 5], 1u << (d & 31));
            }
            __syncthreads();
            // a thread's words, then the sums of the threads before it
            const uint32_t per = (words + EX_THREADS - 1) / EX_THREADS, i0 = threadIdx.x * per;
            uint32_t n = 0;
            for (uint32_t i = i0; i < min(i0 + per, words); ++i) n += __popc(table[i]);
            uint32_t upto = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xffffffffu, upto, o);
                if ((threadIdx.x & 31) >= o) upto += v;
            }
            if ((threadIdx.x & 31) == 31) sum[threadIdx.x >> 5] = upto;
            __syncthreads();
            uint32_t before = upto - n, total = 0;
            for (uint32_t i = 0; i < EX_THREADS / 32; ++i) {
                if (i < threadIdx.x >> 5) before += sum[i];
                total += sum[i];
            }
            chunk[threadIdx.x] = before;
            __syncthreads();
            if (on && sg.x == e.x && sg.y && g >= w0) {
                const uint32_t d = g - w0, word = d >> 5;
                if (word >= words) {
                    rank += total;
                } else {
                    rank += chunk[word / per] + __popc(table[word] & ((1u << (d & 31)) - 1u));
                    for (uint32_t i = word / per * per; i < word; ++i) rank += __popc(table[i]);
                }
            }
            __syncthreads();
        }
    });
    segment_tiles(
        sg.y < EX_WIDE ? sg : make_uint2(0, 0), [&](uint32_t q0, uint32_t n) {
            for (uint32_t q = threadIdx.x; q < n; q += EX_THREADS) s_g[q] = list.entry[q0 + q];
        },
        [&](uint32_t first, uint32_t last) {
#pragma unroll 8
            for (uint32_t q = first; q < last; ++q) rank += s_g[q] < g;
        });
    if (!on) return;
    const uint32_t L = (uint32_t)(t * list.leaves_per_tree) + leaf;
    const int64_t s = reservoir_slot(L, res_count[L] - sg.y + rank, kappa, k0, k1);
    slot[r] = s < 0 ? kNoSlot : (uint16_t)s;
}

__global__ void __launch_bounds__(EX_THREADS) k_adapt_insert(const uint16_t *__restrict__ ex_leaf,
                                                             const uint16_t *__restrict__ slot, ExList list,
                                                             const float4 *__restrict__ ex_pt,
                                                             const uint32_t *__restrict__ res_count, int kappa,
                                                             float4 *__restrict__ res) {
    __shared__ uint2 s_gs[EX_TILE];
    __shared__ uint32_t table[EX_TABLE];
    const int P = list.P, t = blockIdx.y;
    const uint32_t r0 = (uint32_t)t * P + blockIdx.x * EX_THREADS, r = r0 + threadIdx.x, end = list.end(t);
    if (r0 >= end) return;
    const uint32_t g = r < end ? list.entry[r] : 0, mine = r < end ? slot[r] : kNoSlot;
    const uint32_t leaf = r < end ? ex_leaf[(size_t)t * P + g] : 0, L = (uint32_t)(t * list.leaves_per_tree) + leaf;
    const bool on = mine != kNoSlot;
    uint2 sg = r < end ? list.segment(t, leaf) : make_uint2(0, 0);
    if (sg.y && res_count[L] <= (uint32_t)kappa) sg = make_uint2(0, 0);  // every example has a slot of its own
    bool later = false;
    wide_segments(sg, min(end - r0, (uint32_t)EX_THREADS), [&](uint2 e) {
        for (int i = threadIdx.x; i < kappa; i += EX_THREADS) table[i] = 0;
        __syncthreads();
        for (uint32_t q = threadIdx.x; q < e.y; q += EX_THREADS) {
            const uint32_t s = slot[e.x + q];
            if (s != kNoSlot) atomicMax(&table[s], list.entry[e.x + q] + 1);
        }
        __syncthreads();
        if (on && sg.x == e.x && sg.y) later = table[mine] != g + 1;
        __syncthreads();
    });
    segment_tiles(
        on && sg.y < EX_WIDE ? sg : make_uint2(0, 0), [&](uint32_t q0, uint32_t n) {
            for (uint32_t q = threadIdx.x; q < n; q += EX_THREADS)
                s_gs[q] = make_uint2(list.entry[q0 + q], slot[q0 + q]);
        },
        [&](uint32_t first, uint32_t last) {
#pragma unroll 8
            for (uint32_t q = first; q < last; ++q) later |= s_gs[q].x > g && s_gs[q].y == mine;
        });
    if (on && !later) res[(size_t)L * kappa + mine] = ex_pt[g];
}

rl_status adapt_frame(rl_forest *f, const float *depth, const uint8_t *rgb,
                      const rl_intrinsics *K, const double T[16], cudaStream_t s) {
    const rl_forest_params &p = f->p;
    const int o = p.grid_origin, st = p.grid_step;
    const int gw = K->width > o ? (K->width - o + st - 1) / st : 0;
    const int gh = K->height > o ? (K->height - o + st - 1) / st : 0;
    const int P = gw * gh;
    if (P == 0) return RL_OK;
    if (f->ex_capacity < P) {
        arena_free(f->ctx, f->ex_leaf);
        arena_free(f->ctx, f->ex_pt);
        arena_free(f->ctx, f->ex_list);
        f->ex_leaf = nullptr;
        f->ex_pt = nullptr;
        f->ex_list = nullptr;
        f->ex_capacity = 0;
        RL_TRY(alloc_n(f->ctx, (uint64_t)P * p.n_trees * 2, &f->ex_leaf));
        RL_TRY(alloc_n(f->ctx, (uint64_t)P, &f->ex_pt));
        RL_TRY(alloc_n(f->ctx, (uint64_t)P * p.n_trees, &f->ex_list));
        f->ex_capacity = P;
    }
    Pose12 pose;
    for (int i = 0; i < 12; ++i) pose.m[i] = T[i];
    const uint32_t k0 = (uint32_t)f->seed, k1 = (uint32_t)(f->seed >> 32);
    const dim3 grid((P + EX_THREADS - 1) / EX_THREADS, p.n_trees);
    const ExList list{f->ex_list, f->frame_cnt, P, f->leaves_per_tree};
    RL_CK(cudaMemsetAsync(f->frame_cnt, 0, sizeof(uint32_t) * f->n_leaves, s));
    k_adapt_examples<<<grid, EX_THREADS, 0, s>>>(f->nodes, f->n_branch, p.depth, f->leaves_per_tree, depth, rgb, K->width,
                                          K->height, K->fx, K->fy, K->cx, K->cy, pose, gw, gh, st, o, f->ex_leaf,
                                          f->ex_pt, f->frame_cnt);
    RL_LAUNCH_CK();
    const int groups = (f->leaves_per_tree + EX_SCAN_EACH - 1) / EX_SCAN_EACH;  // leaves of a thread
    const int scan = std::min(EX_SCAN_THREADS, (groups + 31) / 32 * 32);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((groups + scan - 1) / scan, p.n_trees);
    cfg.blockDim = dim3(scan);
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cfg.gridDim.x;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    RL_CK(cudaLaunchKernelEx(&cfg, k_adapt_segments, f->frame_cnt, f->res_count, f->leaves_per_tree, P));
    k_adapt_scatter<<<grid, EX_THREADS, 0, s>>>(f->ex_leaf, P, f->leaves_per_tree, f->frame_cnt, f->ex_list);
    RL_LAUNCH_CK();
    uint16_t *slot = f->ex_leaf + (size_t)P * p.n_trees;
    k_adapt_slots<<<grid, EX_THREADS, 0, s>>>(f->ex_leaf, list, f->res_count, p.kappa, k0, k1, slot);
    RL_LAUNCH_CK();
    k_adapt_insert<<<grid, EX_THREADS, 0, s>>>(f->ex_leaf, slot, list, f->ex_pt, f->res_count, p.kappa, f->res);
    RL_LAUNCH_CK();
    return RL_OK;
}

rl_status reset_leaves(rl_forest *f, cudaStream_t s) {
    RL_CK(cudaMemsetAsync(f->res_count, 0, sizeof(uint32_t) * f->n_leaves, s));
    RL_CK(cudaMemsetAsync(f->frame_cnt, 0, sizeof(uint32_t) * f->n_leaves, s));
    RL_CK(cudaMemsetAsync(f->nmodes, 0, f->n_leaves, s));
    RL_CK(cudaMemsetAsync(f->centroid, 0, sizeof(float4) * f->n_leaves, s));
    f->cursor = 0;
    return RL_OK;
}

}  // namespace rl
