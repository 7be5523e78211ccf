// Launch shape of the LM cluster kernel: how many sets of CTAs split a
// frame's hypotheses.  Host code without CUDA.
#pragma once

namespace rl {

// Whole clusters of each shape with more than one set that the GPU holds at
// once, one CTA per SM (0: a cluster of that size does not fit any of its
// GPCs, or is not allowed).
struct LmResident {
    int first4 = 0;  // first round, 4 CTAs on the pixels, 4 sets
    int first2 = 0;  // first round, 2 sets
    int later2 = 0;  // later rounds, 8 CTAs on the pixels, 2 sets
};

// Sets for a call of `frames` frames at work: the most whose clusters are
// resident together, and 1 (clusters of 4 or 8 CTAs, two CTAs per SM) when
// they would queue.  Which GPCs a device has decides what it holds: a GB300
// was seen to hold 7 clusters of 16 CTAs and 15 of 8.  Measured with 25 modes
// per pixel, 8 frames of 640x480, time of the call against one set: 4 sets in
// the first round and 2 later, one cluster waiting, 1.04 (Euclidean distances
// 1.16); 2 in the first round alone 0.96 (0.99); 7 frames, 4 and 2, 0.90
// (0.98).
//
// heavy: 48 modes per pixel or more at Mahalanobis distances.  One cluster may
// then wait, and starts as soon as the shortest of the others ends: 8 frames
// of 50 modes 0.83 (4 and 2 sets; 0.92 without waiting), 16 frames 0.95 (2 and
// 1 sets); where all frames take equally long 1.02 to 1.06.
//
// sparse: a later level of a cascade, where most frames are empty, but all may
// be at work.  Heavy clusters of 16 are then used up to two deep, of 8 up to
// three.  Cascades of 640x480 frames of which one in ten goes on, of 16, 32,
// 48 and 64 frames: 2.08, 2.35, 2.78 and 3.17 ms (2.24, 2.52, 2.88 and 3.21
// with sets for all frames alike, 2.08, 2.31, 2.79 and 3.08 with sets for a
// quarter); with all going on 7.9, 10.4, 13.4 and 16.8 ms (7.5, 10.4, 12.8 and
// 16.9; 7.9, 12.7, 13.3 and 18.4).
inline int lm_sets(const LmResident &r, bool first_round, int frames, bool sparse, bool heavy) {
    auto fits = [&](int held, int deep) {
        return held > 0 && frames <= (heavy ? (sparse ? deep : 1) * (held + 1) : held);
    };
    if (first_round) return fits(r.first4, 2) ? 4 : fits(r.first2, 3) ? 2 : 1;
    return fits(r.later2, 2) ? 2 : 1;
}

}  // namespace rl
