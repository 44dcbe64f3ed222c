// Register-tile kernels: 2D, radius 4, every storage type, both coefficient forms.
#include "tile.h"
#include "tile_kernel.cuh"

namespace stn {
namespace {
const TileEntry kList[] = {
    STN_T4(4, 4, 8),
    STN_T4(4, 8, 8),
    STN_T4(4, 16, 4)};
}  // namespace
int list_tile_r4(const TileEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
