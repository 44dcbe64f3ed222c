// Bounds-checked register tiles (stencil_set_checked): both coefficient forms, 16-bit storage and each tile shape, on
// radii that exchange fewer and as many rows as a warp holds.
#include "tile.h"
#include "tile_kernel.cuh"

namespace stn {
namespace {
const TileEntry kList[] = {STN_TC(1, 4, 8, float, 0, false, true),           STN_TC(3, 8, 8, float, 0, false, true),
                           STN_TC(4, 16, 4, __nv_bfloat16, 1, false, true),  STN_TC(2, 16, 4, float, 0, true, true),
                           STN_TC(6, 8, 8, float, 0, false, true)};
}  // namespace
int list_tile_checked(const TileEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
