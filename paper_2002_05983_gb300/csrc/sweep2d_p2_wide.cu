// Streaming-kernel instantiations: 2D, two rows per step for radius 5 and 6 (every storage type; the
// rule's choice), and four rows per step for radius 3 at t = 2, which the rule's passes over large
// FP32 grids run.  Measured on 16384^2, t = 2, us per step: radius 5 one row / two FP32 410 / 381, BF16
// 486 / 393; radius 6 FP32 639 / 568; radius 3 two rows / four FP32 206.8 / 193.1.
#include "registry.h"
#include "sweep_kernel.cuh"

namespace stn {
namespace {
const KernelEntry kList[] = {
    STN_EP(2, 5, 1, float, 0, 2),
    STN_EP(2, 5, 2, float, 0, 2),
    STN_EP(2, 6, 1, float, 0, 2),
    STN_EP(2, 6, 2, float, 0, 2),
    STN_EP(2, 5, 1, __nv_bfloat16, 1, 2),
    STN_EP(2, 5, 2, __nv_bfloat16, 1, 2),
    STN_EP(2, 6, 1, __nv_bfloat16, 1, 2),
    STN_EP(2, 6, 2, __nv_bfloat16, 1, 2),
    STN_EP(2, 5, 1, __half, 2, 2),
    STN_EP(2, 5, 2, __half, 2, 2),
    STN_EP(2, 6, 1, __half, 2, 2),
    STN_EP(2, 6, 2, __half, 2, 2),
    STN_EP(2, 3, 2, float, 0, 4)};
}  // namespace
int list_2d_p2_wide(const KernelEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
