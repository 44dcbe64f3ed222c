// Table of compiled register-tile kernels (filled by tile2d_*.cu).
#pragma once
#include <cstddef>

#include "sweep_cfg.h"

namespace stn {

struct TileEntry {
    int r, dtype, sh;      // radius; 0 fp32, 1 bf16, 2 fp16; 1: one coefficient per distance
    int v, w;              // rows per thread, warps per block: regions of 128 x (v*w) cells
    size_t smem;           // dynamic shared memory bytes
    const void *fn;        // __global__ tile2d_kernel<r, v, w, S, sh, chk>
    int chk;               // 1: bounds-checked
};

int list_tile_r1(const TileEntry **e);
int list_tile_r2(const TileEntry **e);
int list_tile_r3(const TileEntry **e);
int list_tile_r4(const TileEntry **e);
int list_tile_r5(const TileEntry **e);
int list_tile_r6(const TileEntry **e);
int list_tile_checked(const TileEntry **e);

}  // namespace stn

#define STN_T(R, V, W, S, DT, SH) STN_TC(R, V, W, S, DT, SH, false)
#define STN_TC(R, V, W, S, DT, SH, CHK)                                                               \
    {R, DT, (SH) ? 1 : 0, V, W, stn::TileGeo<R, V, W>::SMEM,                                          \
     reinterpret_cast<const void *>(&stn::tile2d_kernel<R, V, W, S, SH, CHK>), (CHK) ? 1 : 0}
#define STN_T4(R, V, W)                                                                               \
    STN_T(R, V, W, float, 0, false), STN_T(R, V, W, __nv_bfloat16, 1, false),                         \
        STN_T(R, V, W, __half, 2, false), STN_T(R, V, W, float, 0, true)
