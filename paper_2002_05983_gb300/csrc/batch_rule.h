// Which form a batch takes (host code without CUDA types).
#pragma once
#include <algorithm>
#include <cstdint>

namespace stn {

// Graphs of per-grid chains have one node per pass; longer lists keep the persistent launches, whose
// size does not grow with the steps.
constexpr int64_t kMaxChainNodes = 20000;

// Lists with, on average, fewer than this many grids per kernel class (dimension, radius, storage type, coefficient
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

// Blocks of a persistent class: at most the resident slots, the tiles of all its passes, and twice the
// tiles of one pass of every grid.  At most one pass of a grid can run at a time, so more blocks would
// only hold registers and shared memory while they wait, which the classes beside this one need (64
// grids of 64^3, radius 1 to 4: 12.4-15.4 -> 7.9 ms); once the pass's tiles alone are allowed, blocks waiting for a
// slow grid keep ready tiles of the next pass from being taken (64 of 1024^2: 14.1 ms with every slot or
// twice the tiles, 15.6 with the tiles).  Over 147 lists 0.90 of the time with every slot, none slower.
inline int64_t batch_blocks(int64_t tiles, int64_t pass_tiles, int64_t slots)
{
    return std::min(std::min(tiles, 2 * pass_tiles), slots);
}

}  // namespace stn
