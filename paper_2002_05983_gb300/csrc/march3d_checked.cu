// Bounds-checked marching kernels (stencil_set_checked), with vector loads and cell by cell.
#include "march.h"
#include "march_kernel.cuh"

namespace stn {
namespace {
const MarchEntry kList[] = {STN_MC(1, float, 0, false, true), STN_MC(4, float, 0, false, true), STN_MC(3, __half, 2, false, true),
                            STN_MC(2, float, 0, true, true)};
}  // namespace
int list_march_checked(const MarchEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
