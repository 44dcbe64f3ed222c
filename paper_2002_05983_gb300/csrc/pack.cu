// Copies a grid with rows of any length and alignment into one whose rows start on 16-byte
// boundaries, the cells between a row's end and the next whole 4-cell vector repeating its last
// cell: the layout that the kernels for rows of any length read.  Bound by memory; one pass over
// the grid once per run (251 x 243 x 237 FP32: the copy and one pass of two steps 63 us, every further pass 36.5).
//
// Launched as a programmatic dependent, so its blocks may be resident while the work before it in
// the stream still writes `in`: the pointers carry no __restrict__, which with const would let the
// loads go through the read-only path or ahead of grid_dep_wait.
#include "pack.h"

#include "sweep_kernel.cuh"

namespace stn {
namespace {

template <typename W>
__global__ void __launch_bounds__(256) pack_kernel(const W *in, W *out, int nx, int pitch, int64_t rows)
{
    grid_dep_launch();
    grid_dep_wait();
    const int nv = (nx + 3) / 4;
    for (int64_t r = static_cast<int64_t>(blockIdx.x) * 8 + threadIdx.y; r < rows; r += static_cast<int64_t>(gridDim.x) * 8) {
        const W *src = in + r * nx;
        W *dst = out + r * pitch;
        for (int v = threadIdx.x; v < nv; v += 32) {
            W e[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) e[c] = src[min(4 * v + c, nx - 1)];
            if constexpr (sizeof(W) == 4)
                *reinterpret_cast<uint4 *>(dst + 4 * v) = make_uint4(e[0], e[1], e[2], e[3]);
            else
                *reinterpret_cast<uint2 *>(dst + 4 * v) =
                    make_uint2(static_cast<uint32_t>(e[0]) | (static_cast<uint32_t>(e[1]) << 16),
                               static_cast<uint32_t>(e[2]) | (static_cast<uint32_t>(e[3]) << 16));
        }
    }
}

}  // namespace

const void *pack_fn(int elem_bytes)
{
    return elem_bytes == 4 ? reinterpret_cast<const void *>(&pack_kernel<uint32_t>)
                           : reinterpret_cast<const void *>(&pack_kernel<uint16_t>);
}

}  // namespace stn
