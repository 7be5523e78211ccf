// Launch shape of the ICP kernels: blocks per pose.  Host code without CUDA.
#pragma once

#include <stdint.h>

namespace rl {

// Whole clusters of 8 and of 4 blocks that the GPU holds at once.
struct IcpResident {
    int of8 = 0, of4 = 0;
};

// Blocks per pose (8, 4 or 1) for `poses` poses at work, an iteration
// evaluating `cells` pixels on average (strides included).  A cluster must be
// resident beside all others, and a pose must have the pixels to pay for two
// cluster barriers an iteration, the more the more blocks an SM shares.
// Measured with the default levels (an iteration evaluates 0.284 of the
// image); microseconds a call with one, four and eight blocks per pose:
//   16 poses: 160x120 267, 293, 292; 240x180 319, 318, 306; 640x480 899, 667,
//   496; 50 poses: 240x180 321, 346, 333; 320x240 386, 394, 360; 64 poses:
//   320x240 386, 396, 594; 400x300 484, 457, 667; 100 poses: 400x300 487, 496;
//   500x375 637, 618; 136 poses: 500x375 641, 683; 640x480 898, 930, but
//   calls of 8 and 9 frames with ICP 3.89 and 4.11 ms, 3.62 and 3.77 with
//   four: poses outside the box take longer per pixel.  152 poses, of which a
//   GB300 does not hold all clusters of four: 640x480 908, 1403.
inline int icp_blocks(const IcpResident &r, int sm_count, int64_t poses, double cells) {
    auto load = [&](int c) { return (poses * c + sm_count - 1) / sm_count; };  // blocks on an SM
    if (poses <= r.of8 && cells >= (load(8) <= 2 ? 12e3 : 20e3)) return 8;
    if (poses <= r.of4 && cells >= (load(4) <= 2 ? 34e3 : load(4) == 3 ? 53e3 : 85e3)) return 4;
    return 1;
}

}  // namespace rl
