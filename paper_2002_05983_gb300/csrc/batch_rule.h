// Which form a batch takes (host code without CUDA types).
#pragma once
#include <cstdint>

namespace stn {

// Graphs of per-grid chains have one node per pass; longer lists keep the persistent launches, whose
// size does not grow with the steps.
constexpr int64_t kMaxChainNodes = 20000;

// Lists with fewer than this many grids per kernel class (dimension, radius, storage type, coefficient
// form) run as chains.  A persistent class advances all its grids side by side, one tile latency (25-50
// us) a pass however few they are, and holds its blocks' SMs until it ends; chains take each grid's own
// fastest passes, but 2D grids one after another, and their graph costs 3-5 us a pass to build.
// Measured over 346 lists of 2 to 64 grids in 1 to 8 classes (2D sides 128-4096, 3D sides 32-320, 10 to
// 1000 steps): below three grids per class chains take 0.08-0.90 of the persistent launches' time; from
// three on 0.3-2.4 (100 steps: 47 grids of 256^2 radius 1 3.5 against 1.5 ms, 32 of 64^3 radius 4 9.2 against 5.6, 16
// of 128^3 radius 1 7.0 against 3.9), and a first call on new buffers up to 4 times as long.
constexpr int kClassGrids = 3;

inline bool batch_as_chains(int grids, int classes, int64_t passes)
{
    return grids < kClassGrids * classes && passes <= kMaxChainNodes;
}

}  // namespace stn
