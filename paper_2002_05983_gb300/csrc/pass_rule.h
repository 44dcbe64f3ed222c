// How a streaming pass is launched (host code without CUDA types).
#pragma once
#include <cstdint>

namespace stn {

// Whether a 3D streaming pass is launched as a programmatic dependent of the pass before it: where its
// segments fill whole waves, or its blocks the device's slots five quarters times, and the pass before is
// of the same kind (or the copy that pads rows, which fills the device).  Blocks launched beside a smaller
// pass would take the slots that the pass before leaves free, several on one SM while others have none.
// Time with dependent launches over time without, 630 (kernel, shape) pairs of one schedule each: below a
// quarter of a wave 0.97 on average and up to 1.38 (radius 3 64 x 64 x 2000), from there to a half 1.12
// (1.32), to three quarters 1.05 (1.23), to one 0.97 (1.19), to five quarters 0.96 (1.07), above 0.96 (1.01).
// A remainder pass and the run after it: radius 1 154 x 653 x 368, 3 steps a call 135.8 -> 122.1 us.
inline bool dependent_pass(bool whole_waves, int64_t blocks, int64_t slots) { return whole_waves || 4 * blocks >= 5 * slots; }

}  // namespace stn
