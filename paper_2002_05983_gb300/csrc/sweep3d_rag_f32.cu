// Streaming-kernel instantiations for rows of any length (3D, float storage, radius 1..3): the degrees and rows per
// thread or step that the library's rule uses.
#include "registry.h"
#include "sweep_kernel.cuh"

namespace stn {
namespace {
const KernelEntry kList[] = {
    STN_ER(3, 1, 1, 2, float, 0, false, 1),
    STN_ER(3, 1, 2, 2, float, 0, false, 1),
    STN_ER(3, 2, 1, 2, float, 0, false, 1),
    STN_ER(3, 3, 1, 4, float, 0, false, 1),
    STN_ER(3, 1, 1, 2, float, 0, true, 1),
    STN_ER(3, 1, 2, 2, float, 0, true, 1),
    STN_ER(3, 2, 1, 2, float, 0, true, 1)};
}  // namespace
int list_rag_f32(const KernelEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
