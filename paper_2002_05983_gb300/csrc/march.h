// Table of compiled marching kernels (filled by march3d_*.cu).
#pragma once

namespace stn {

struct MarchEntry {
    int r, dtype, sh;   // radius; 0 fp32, 1 bf16, 2 fp16; 1: one coefficient per distance
    int vec;            // 1: vector loads (input rows start on whole 4-cell vectors)
    const void *fn;     // __global__ march3d_kernel<r, S, sh, vec, chk>
    int chk;            // 1: bounds-checked
};

int list_march_r1(const MarchEntry **e);
int list_march_r2(const MarchEntry **e);
int list_march_r3(const MarchEntry **e);
int list_march_r4(const MarchEntry **e);
int list_march_checked(const MarchEntry **e);

}  // namespace stn

#define STN_M(R, S, DT, SH) STN_MC(R, S, DT, SH, false)
#define STN_MC(R, S, DT, SH, CHK)                                                                             \
    {R, DT, (SH) ? 1 : 0, 1, reinterpret_cast<const void *>(&stn::march3d_kernel<R, S, SH, true, CHK>), (CHK) ? 1 : 0},    \
        {R, DT, (SH) ? 1 : 0, 0, reinterpret_cast<const void *>(&stn::march3d_kernel<R, S, SH, false, CHK>), (CHK) ? 1 : 0}
