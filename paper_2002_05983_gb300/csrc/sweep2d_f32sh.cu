// Streaming-kernel instantiations with one coefficient per distance (shared
// coefficients), float storage; 2D, 128 threads x 4 cells per block row,
// radius 1..4 at the temporal degrees the full-coefficient defaults use, for radius 2..4 with one
// and with two rows per step (the rule's choice: 16384^2 us per step, one row / two: radius 2 169.3 /
// 151.9, 3 246 / 218, 4 301 / 247).
#include "registry.h"
#include "sweep_kernel.cuh"

namespace stn {
namespace {
const KernelEntry kList[] = {
    STN_EX(2, 1, 1, 1, float, 0, 128, 1, true),
    STN_EX(2, 1, 2, 1, float, 0, 128, 1, true),
    STN_EX(2, 1, 3, 1, float, 0, 128, 1, true),
    STN_EX(2, 1, 4, 1, float, 0, 128, 1, true),
    STN_EX(2, 1, 5, 1, float, 0, 128, 1, true),
    STN_EX(2, 2, 1, 1, float, 0, 128, 1, true),
    STN_EX(2, 2, 2, 1, float, 0, 128, 1, true),
    STN_EX(2, 2, 3, 1, float, 0, 128, 1, true),
    STN_EX(2, 3, 1, 1, float, 0, 128, 1, true),
    STN_EX(2, 3, 2, 1, float, 0, 128, 1, true),
    STN_EX(2, 4, 1, 1, float, 0, 128, 1, true),
    STN_EX(2, 4, 2, 1, float, 0, 128, 1, true),
    STN_EXC(2, 2, 1, 1, float, 0, 128, 1, true, false, 2),
    STN_EXC(2, 2, 2, 1, float, 0, 128, 1, true, false, 2),
    STN_EXC(2, 2, 3, 1, float, 0, 128, 1, true, false, 2),
    STN_EXC(2, 3, 1, 1, float, 0, 128, 1, true, false, 2),
    STN_EXC(2, 3, 2, 1, float, 0, 128, 1, true, false, 2),
    STN_EXC(2, 4, 1, 1, float, 0, 128, 1, true, false, 2),
    STN_EXC(2, 4, 2, 1, float, 0, 128, 1, true, false, 2)};
}  // namespace
int list_2d_f32sh(const KernelEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
