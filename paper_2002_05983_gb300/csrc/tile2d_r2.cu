// Register-tile kernels: 2D, radius 2, every storage type, both coefficient forms.
#include "tile.h"
#include "tile_kernel.cuh"

namespace stn {
namespace {
const TileEntry kList[] = {
    STN_T4(2, 4, 8),
    STN_T4(2, 8, 8),
    STN_T4(2, 16, 4)};
}  // namespace
int list_tile_r2(const TileEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
