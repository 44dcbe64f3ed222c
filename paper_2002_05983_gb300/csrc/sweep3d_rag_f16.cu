// Streaming-kernel instantiations for rows of any length (3D, __half storage, rounded at every step): the degrees and rows per
// thread or step that the library's rule uses.
#include "registry.h"
#include "sweep_kernel.cuh"

namespace stn {
namespace {
const KernelEntry kList[] = {
    STN_ER(3, 1, 1, 2, __half, 2, false, 1),
    STN_ER(3, 2, 1, 4, __half, 2, false, 1),
    STN_ER(3, 3, 1, 4, __half, 2, false, 1),
    STN_ER(3, 4, 1, 4, __half, 2, false, 1),
    STN_ER(3, 5, 1, 2, __half, 2, false, 1),
    STN_ER(3, 6, 1, 2, __half, 2, false, 1)};
}  // namespace
int list_rag_f16(const KernelEntry **e)
{
    *e = kList;
    return static_cast<int>(sizeof(kList) / sizeof(kList[0]));
}
}  // namespace stn
