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
// resident together, all but one, and 1 (clusters of 4 or 8 CTAs, two CTAs
// per SM) when more would queue.  Which GPCs a device has decides what it
// holds: a GB300 was seen to hold 7 clusters of 16 CTAs and 15 of 8.  The one
// cluster that may wait starts as soon as the shortest of the others ends:
// there a call of 8 frames of 640x480 takes 3.90 ms (4.32 with half the
// sets), one of 16 frames 5.33 (5.60 with one set).
inline int lm_sets(const LmResident &r, bool first_round, int frames) {
    auto fits = [frames](int held) { return held > 0 && frames <= held + 1; };
    if (first_round) return fits(r.first4) ? 4 : fits(r.first2) ? 2 : 1;
    return fits(r.later2) ? 2 : 1;
}

}  // namespace rl
