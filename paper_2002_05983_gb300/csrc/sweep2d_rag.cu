// Streaming-kernel instantiations for rows of any length (2D, float storage, the radii that large grids stream): the degrees and rows per
// thread or step that the library's rule uses.
#include "registry.h"
#include "sweep_kernel.cuh"

namespace stn {
namespace {
const KernelEntry kList[] = {
    STN_ER(2, 2, 1, 1, float, 0, false, 2),
    STN_ER(2, 2, 2, 1, float, 0, false, 2),
    STN_ER(2, 2, 3, 1, float, 0, false, 2),
    STN_ER(2, 3, 1, 1, float, 0, false, 2),
    STN_ER(2, 3, 2, 1, float, 0, false, 2),
    STN_ER(2, 4, 1, 1, float, 0, false, 2),
    STN_ER(2, 4, 2, 1, float, 0, false, 2),
    STN_ER(2, 5, 1, 1, float, 0, false, 2),
    STN_ER(2, 5, 2, 1, float, 0, false, 2)};
}  // namespace
int list_rag_2d(const KernelEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
