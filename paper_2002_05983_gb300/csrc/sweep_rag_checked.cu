// Bounds-checked streaming kernels for rows of any length (stencil_set_checked): both dimensions, both storage
// widths, one and two levels (rows per thread and step of a checked handle's schedule).
#include "registry.h"
#include "sweep_kernel.cuh"

namespace stn {
namespace {
const KernelEntry kList[] = {
    STN_ERC(3, 1, 1, 2, float, 0, false, true, 1), STN_ERC(3, 1, 2, 2, float, 0, false, true, 1),
    STN_ERC(3, 4, 1, 2, float, 0, false, true, 1), STN_ERC(3, 2, 1, 2, __half, 2, false, true, 1),
    STN_ERC(2, 4, 1, 1, float, 0, false, true, 1), STN_ERC(2, 4, 2, 1, float, 0, false, true, 1)};
}  // namespace
int list_rag_checked(const KernelEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
