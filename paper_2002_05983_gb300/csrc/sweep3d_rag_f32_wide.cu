// Streaming-kernel instantiations for rows of any length (3D, float storage, radius 4..6 and radius 3, 4 with one coefficient per distance): the degrees and rows per
// thread or step that the library's rule uses.
#include "registry.h"
#include "sweep_kernel.cuh"

namespace stn {
namespace {
const KernelEntry kList[] = {
    STN_ER(3, 4, 1, 4, float, 0, false, 1),
    STN_ER(3, 5, 1, 4, float, 0, false, 1),
    STN_ER(3, 6, 1, 2, float, 0, false, 1),
    STN_ER(3, 3, 1, 2, float, 0, true, 1),
    STN_ER(3, 4, 1, 2, float, 0, true, 1)};
}  // namespace
int list_rag_f32_wide(const KernelEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
