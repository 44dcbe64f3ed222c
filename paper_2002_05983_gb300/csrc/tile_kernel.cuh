// Register-tile sweep of 2D grids for sm_103a: t time steps of one tile per block, the tile
// held in registers.
//
// A block of W warps owns a region of 128 x (W*V) cells: lane l of warp w keeps cells
// 4l..4l+3 of rows w*V .. w*V + V-1, so a warp spans the region's width and every load and
// store of a row is 512 contiguous bytes.  One step of all rows is
//   * x neighbours: r shuffles per side and row (4 cells each);
//   * y neighbours: the thread's own registers, and the r rows beyond its V from the warps
//     above and below through shared memory (double-buffered, one barrier per step);
//   * one multiply and 2*D*r FMAs per cell in Eq. 1's order, so the bits are those of every
//     other schedule.
// The valid part shrinks by r cells per step (overlapped temporal blocking, Eq. 2): regions
// overlap by h = r*t rows and hx = h rounded up to 4 columns per side.
//
// Against the streaming kernel (sweep_kernel.cuh) a step needs no copy wait, no ring
// addressing and no per-row bookkeeping, and the loop over t is a loop: the code is one step of
// one tile whatever the degree, which the instruction cache holds, and a pass of any degree
// runs on the same kernel.  The price is the halo in y as well as in x.
//
// What bounds it: the issue slots (0.62 per scheduler; FFMA and FMUL 64-72 % of the instructions at
// one cell per instruction, packed pairs now take half the slots of the y terms and of the even x
// terms: 16384^2 radius 1 t = 8 942 -> 780 us, radius 4 t = 2 919 -> 699 us) and the load phase of
// each tile, which the other resident blocks cover.  Small grids are bound by latency: a step of
// a lone block takes 0.45 us with 4 rows per thread, 0.7 us with 8.  Hence three shapes: 8 warps x
// 4 rows for grids that leave SMs idle otherwise (256^2: 0.7 against 0.9 us per step), 8 x 8 for
// the middle, 4 x 16 where there are many tiles (fewest exchanged rows; 16384^2 radius 1 2745
// against 2261 GCell/s with 8 x 8).  Wider blocks (16 warps, 12 rows, 256-row regions) measured
// 4-30 % slower.
//
// Passes are launched as programmatic dependents: the next pass's blocks are placed while the last
// blocks of this one run and wait for its end before they read (256^2, radius 1, t = 4: 6.2 -> 3.4
// us per pass).
//
// Clamp to edge: rows above the grid are never in a region (tile rows start at 0); the first
// warp's rows above are copies of its row 0.  Columns left and right of the grid and rows below
// it lie in the region of edge tiles and take the border cell's value after every step
// (fix_edges, block-uniform branches that interior tiles skip).  Nothing assumes whole vectors:
// rows of any length and base address run, with vector loads and stores where they are aligned.
// Between the passes of a run, rows of any length sit at 16-byte pitches, so only the first pass
// loads and the last pass stores cell by cell (3001 x 2047, radius 3, 50 steps: 514 -> 410 us).
#pragma once

#include "sweep_kernel.cuh"

namespace stn {

constexpr int kTileW = 128;          // region width in cells: one warp, 4 cells per lane
constexpr int kMaxK2 = 4 * kMaxR + 1;

struct TileArgs {
    const void *in;
    void *out;
    int nx, ny;
    int pin, pout;        // row pitches (cells)
    int t;                // steps of this pass
    int rnd;              // 16-bit storage: round to the storage type after every rnd steps
    int h, hx;            // halo rows r*t and halo columns (a multiple of 4)
    int ntx;              // tiles per tile row
    int vin, vout;        // rows start on whole 4-cell vectors: vector loads / stores
    float c[kMaxK2];
    unsigned *status;     // bounds-checked kernels: device status word
};

template <int R, int V, int W> struct TileGeo {
    static constexpr int TH = W * V;                             // region rows
    static constexpr int NB = V < 2 * R ? V : 2 * R;             // rows a warp hands to its neighbours
    static constexpr size_t SMEM = sizeof(float4) * 2 * W * NB * 32;
    static_assert(V >= R, "a warp's neighbour rows come from one warp per side");
};

__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// rounds to the storage type and back (the value a pass boundary would store)
template <typename S> __device__ __forceinline__ void round4(float (&v)[4])
{
    if constexpr (sizeof(S) == 2) {
        S tmp[4] __attribute__((aligned(8)));
        Fmt<S>::store4(tmp, v);
        Fmt<S>::load4(tmp, v);
    }
}

template <typename S> __device__ __forceinline__ float cell_in(const S *p);
template <> __device__ __forceinline__ float cell_in<float>(const float *p) { return *p; }
template <> __device__ __forceinline__ float cell_in<__nv_bfloat16>(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
template <> __device__ __forceinline__ float cell_in<__half>(const __half *p) { return __half2float(*p); }

__device__ __forceinline__ float4 f4(const float (&v)[4]) { return make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void set4(float (&v)[4], float4 t) { v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w; }

// Tile `blk` of one pass.  CHK: every global load and store must lie in the rows' cells and every shared-memory
// access in the exchange buffer; one that does not sets kStatusBounds and is skipped.
template <int R, int V, int W, typename S, bool SH, bool CHK, typename A>
__device__ __forceinline__ void tile2d(const A &a, int blk, float4 *halo)
{
    using G = TileGeo<R, V, W>;
    constexpr int NB = G::NB, TH = G::TH;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int bx = blk % a.ntx, by = blk / a.ntx;
    const int ox = bx * (kTileW - 2 * a.hx) - a.hx, oy = by * (TH - 2 * a.h);
    const int gx = ox + 4 * lane, gy0 = oy + w * V;
    const bool live = gy0 < a.ny;                  // warps below the grid only meet the barriers
    const bool below = gy0 + V >= a.ny;            // the next warp's rows are outside the grid
    const bool xedge = ox < 0 || ox + kTileW > a.nx;
    const bool last_y = oy + TH >= a.ny;

    auto ok = [&](int64_t at, int n, int64_t limit) -> bool {
        if constexpr (CHK) {
            if (at >= 0 && at + n <= limit) return true;
            atomicOr(a.status, kStatusBounds);
            return false;
        } else {
            return true;
        }
    };
    auto ok_in = [&](int64_t at, int n) { return ok(at, n, static_cast<int64_t>(a.ny - 1) * a.pin + a.nx); };
    auto ok_out = [&](int64_t at, int n) { return ok(at, n, static_cast<int64_t>(a.ny - 1) * a.pout + a.nx); };
    auto ok_halo = [&](const float4 *p) { return ok(p - halo, 1, 2 * W * NB * 32); };

    float q[V][4];
    if (live) {
        const S *in = static_cast<const S *>(a.in);
        if (a.vin && gx >= 0 && gx + 4 <= a.nx) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int64_t at = static_cast<int64_t>(min(gy0 + v, a.ny - 1)) * a.pin + gx;
                if (ok_in(at, 4)) Fmt<S>::load4(in + at, q[v]);
            }
        } else {
            int xc[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) xc[c] = min(max(gx + c, 0), a.nx - 1);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int64_t row = static_cast<int64_t>(min(gy0 + v, a.ny - 1)) * a.pin;
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (ok_in(row + xc[c], 1)) q[v][c] = cell_in<S>(in + row + xc[c]);
            }
        }
    }

    // out-of-grid columns and rows of the region take the border cell's value
    const int ll = (-ox) >> 2;                                      // lane of x = 0 (cell 0) where ox < 0
    const int lr = (a.nx - 1 - ox) >> 2, cr = (a.nx - 1 - ox) & 3;  // lane and cell of x = nx - 1
    const int vb = a.ny - 1 - gy0;                                  // own row of y = ny - 1
    auto fix_edges = [&]() {
        if (xedge) {
            if (ox < 0) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const float e = __shfl_sync(0xffffffffu, q[v][0], ll);
#pragma unroll
                    for (int c = 0; c < 4; ++c) q[v][c] = lane < ll ? e : q[v][c];
                }
            }
            if (ox + kTileW > a.nx) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const float m = cr == 0 ? q[v][0] : cr == 1 ? q[v][1] : cr == 2 ? q[v][2] : q[v][3];
                    const float e = __shfl_sync(0xffffffffu, m, lr);
#pragma unroll
                    for (int c = 0; c < 4; ++c) q[v][c] = (lane > lr || (lane == lr && c > cr)) ? e : q[v][c];
                }
            }
        }
        if (vb < V - 1) {
#pragma unroll
            for (int v = 1; v < V; ++v)
#pragma unroll
                for (int c = 0; c < 4; ++c) q[v][c] = v > vb ? q[v - 1][c] : q[v][c];
        }
    };

    for (int s = 0;;) {
        float4 *buf = halo + (s & 1) * (W * NB * 32) + lane;
        if (live) {
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (ok_halo(buf + (w * NB + k) * 32)) buf[(w * NB + k) * 32] = f4(q[(NB < 2 * R || k < R) ? k : V - 2 * R + k]);
        }
        __syncthreads();
        ++s;
        // rows that no output of the last step depends on any more are not advanced
        const int dead = R * s;
        const bool need = live && (by == 0 || (w + 1) * V > dead) && (last_y || w * V < TH - dead);
        if (need) {
            float up[R][4], dn[R][4];
#pragma unroll
            for (int m = 0; m < R; ++m) {
                if (w > 0 && ok_halo(buf + ((w - 1) * NB + NB - 1 - m) * 32)) set4(up[m], buf[((w - 1) * NB + NB - 1 - m) * 32]);
                else set4(up[m], f4(q[0]));
                if (!below && w < W - 1 && ok_halo(buf + ((w + 1) * NB + m) * 32)) set4(dn[m], buf[((w + 1) * NB + m) * 32]);
                else set4(dn[m], f4(q[V - 1]));
            }
            auto yn = [&](int y) -> const float * {   // row y of the old field, -R <= y < V + R
                return y < 0 ? up[cclamp(-y - 1, 0, R - 1)] : y >= V ? dn[cclamp(y - V, 0, R - 1)] : q[cclamp(y, 0, V - 1)];
            };
            float n[V][4];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float xl[R], xr[R];   // cells x0 - 1 - k and x0 + 4 + k of this row
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    xl[k] = __shfl_up_sync(0xffffffffu, q[v][3 - (k & 3)], k / 4 + 1);
                    xr[k] = __shfl_down_sync(0xffffffffu, q[v][k & 3], k / 4 + 1);
                }
                auto xn = [&](int x) -> float {   // cell x of this row, -R <= x < 4 + R
                    return x < 0 ? xl[cclamp(-x - 1, 0, R - 1)] : x > 3 ? xr[cclamp(x - 4, 0, R - 1)] : q[v][cclamp(x, 0, 3)];
                };
                // SH: the neighbours at each distance are summed, then one FMA per distance.  Else
                // two cells advance per packed instruction (each lane an IEEE operation of its own,
                // in the same order); their y neighbours and their x neighbours at even distance
                // are register pairs as they stand, x neighbours at odd distance go one by one.
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                    if constexpr (SH) {
                        uint64_t acc = mul2(pk2(a.c[0], a.c[0]), pk2(q[v][c], q[v][c + 1]));
#pragma unroll
                        for (int i = 1; i <= R; ++i) {
                            uint64_t sum;
                            if ((i & 1) == 0) sum = add2(pk2(xn(c - i), xn(c + 1 - i)), pk2(xn(c + i), xn(c + 1 + i)));
                            else sum = pk2(__fadd_rn(xn(c - i), xn(c + i)), __fadd_rn(xn(c + 1 - i), xn(c + 1 + i)));
                            sum = add2(sum, pk2(yn(v - i)[c], yn(v - i)[c + 1]));
                            sum = add2(sum, pk2(yn(v + i)[c], yn(v + i)[c + 1]));
                            acc = fma2(pk2(a.c[i], a.c[i]), sum, acc);
                        }
                        upk2(acc, n[v][c], n[v][c + 1]);
                    } else {
                        uint64_t acc = mul2(pk2(a.c[0], a.c[0]), pk2(q[v][c], q[v][c + 1]));
#pragma unroll
                        for (int i = 1; i <= R; ++i) {
                            const float cw = a.c[4 * i - 3], ce = a.c[4 * i - 2], cs = a.c[4 * i - 1], cn = a.c[4 * i];
                            if ((i & 1) == 0) {
                                acc = fma2(pk2(cw, cw), pk2(xn(c - i), xn(c + 1 - i)), acc);
                                acc = fma2(pk2(ce, ce), pk2(xn(c + i), xn(c + 1 + i)), acc);
                            } else {
                                float a0, a1;
                                upk2(acc, a0, a1);
                                a0 = __fmaf_rn(cw, xn(c - i), a0);
                                a1 = __fmaf_rn(cw, xn(c + 1 - i), a1);
                                a0 = __fmaf_rn(ce, xn(c + i), a0);
                                a1 = __fmaf_rn(ce, xn(c + 1 + i), a1);
                                acc = pk2(a0, a1);
                            }
                            acc = fma2(pk2(cs, cs), pk2(yn(v - i)[c], yn(v - i)[c + 1]), acc);
                            acc = fma2(pk2(cn, cn), pk2(yn(v + i)[c], yn(v + i)[c + 1]), acc);
                        }
                        upk2(acc, n[v][c], n[v][c + 1]);
                    }
                }
            }
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int c = 0; c < 4; ++c) q[v][c] = n[v][c];
        }
        if (s == a.t) break;
        if (need) {
            if constexpr (sizeof(S) == 2) {
                if (s % a.rnd == 0) {
#pragma unroll
                    for (int v = 0; v < V; ++v) round4<S>(q[v]);
                }
            }
            if (xedge || vb < V - 1) fix_edges();
        }
    }

    if (live) {
        const int xl = 4 * lane;
        const int r0 = by == 0 ? 0 : a.h, r1 = last_y ? TH : TH - a.h;   // region rows this tile outputs
        if (xl >= a.hx && xl < kTileW - a.hx && gx < a.nx) {
            S *out = static_cast<S *>(a.out) + static_cast<int64_t>(gy0) * a.pout + gx;
            if (a.vout && gx + 4 <= a.nx) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const int y = w * V + v;
                    if (y >= r0 && y < r1 && gy0 + v < a.ny && ok_out(static_cast<int64_t>(gy0 + v) * a.pout + gx, 4))
                        Fmt<S>::store4(out + static_cast<int64_t>(v) * a.pout, q[v]);
                }
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const int y = w * V + v;
                    if (y >= r0 && y < r1 && gy0 + v < a.ny) {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (gx + c < a.nx && ok_out(static_cast<int64_t>(gy0 + v) * a.pout + gx + c, 1))
                                out[static_cast<int64_t>(v) * a.pout + c] = to_storage<S>(q[v][c]);
                    }
                }
            }
        }
    }
}

// One pass over the grid, one tile per block.
template <int R, int V, int W, typename S, bool SH, bool CHK = false>
__global__ void __launch_bounds__(32 * W, V <= 8 ? 2 : 1) tile2d_kernel(const __grid_constant__ TileArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    grid_dep_launch();
    grid_dep_wait();
    tile2d<R, V, W, S, SH, CHK>(a, static_cast<int>(blockIdx.x), reinterpret_cast<float4 *>(smem));
}

}  // namespace stn
