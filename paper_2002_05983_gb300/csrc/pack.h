#pragma once

namespace stn {

// __global__ pack_kernel<W>(const W *in, W *out, int nx, int pitch, int64_t rows) for 4- or 2-byte
// cells: blocks of 32 x 8 threads, 8 rows each at a time.
const void *pack_fn(int elem_bytes);

}  // namespace stn
