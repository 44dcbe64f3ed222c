// Marching one-step kernels: 3D, radius 1, every storage type, both coefficient forms for FP32,
// with vector loads and cell by cell.
#include "march.h"
#include "march_kernel.cuh"

namespace stn {
namespace {
const MarchEntry kList[] = {STN_M(1, float, 0, false), STN_M(1, __nv_bfloat16, 1, false), STN_M(1, __half, 2, false),
                            STN_M(1, float, 0, true)};
}  // namespace
int list_march_r1(const MarchEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
