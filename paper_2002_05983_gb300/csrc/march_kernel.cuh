// One-step sweep of small 3D grids for sm_103a that marches along z in registers.
//
// A thread owns 4 x cells of a row and a run of z planes.  It keeps the 2r+1 planes around the one
// it computes in registers (a queue that rotates through the unrolled loop, so no moves), loaded one
// plane ahead.  x neighbours come by shuffles within the 16 lanes of a row (the end lanes load
// theirs), y neighbours as whole vectors from the rows next door, which other warps of the block
// loaded r planes earlier: L1 hits.  Nothing is staged in shared memory and no step has a barrier, so a
// run of one to four planes costs no pipeline fill and a 64 x 16 tile gives a block per few planes:
// what a small grid needs to fill 152 SMs.  Bound by latency there (0.4 us a plane for a lone block;
// 64^3 radius 2: 2.8 us a pass, the streaming kernel 4.0; 96^3 radius 4: 5.4 against 9.3), and by L1
// throughput where there are many planes per SM (2r+1 vector loads a cell vector; 256^3 radius 2: 37
// us, streaming 25).  Two rows per thread measured slower at every size (130-180 registers).
#pragma once

#include "tile_kernel.cuh"

namespace stn {

constexpr int kMarchTX = 16, kMarchThreads = 256;   // tiles of 64 x 16 cells

struct MarchArgs {
    const void *in;
    void *out;
    int nx, ny, nz;
    int pin, pout;          // row pitches (cells)
    int seg;                // planes per block
    int ntx, nty;           // tiles in x and y
    int vout;               // 4-cell vector stores
    float c[kMaxK];
    unsigned *status;       // bounds-checked kernels: device status word
};

// V: vector loads (rows start on whole 4-cell vectors); else cell by cell.  CHK: every load must lie in the input's
// rows (to the pitch's end with vectors) and every store in the output's; one that does not sets kStatusBounds
// and is skipped.
template <int R, typename S, bool SH, bool V, bool CHK = false>
__global__ void __launch_bounds__(kMarchThreads) march3d_kernel(const __grid_constant__ MarchArgs a)
{
    static_assert(R <= 4, "one vector of x neighbours per side");
    constexpr int TX = kMarchTX, VY = 1;
    constexpr int PF = 1;                    // planes loaded ahead
    constexpr int Q = 2 * R + 1 + PF;        // queue slots: plane p sits in slot (p - z0 + R) mod Q
    constexpr int GY = kMarchThreads / TX;   // rows of a block
    grid_dep_launch();
    const int tx = threadIdx.x % TX, gr = threadIdx.x / TX;
    const int b = blockIdx.x, cols = a.ntx * a.nty;
    const int bx = b % cols % a.ntx, by = b % cols / a.ntx, bz = b / cols;
    const int gx = bx * 4 * TX + 4 * tx, gy0 = by * GY + gr * VY;
    const int z0 = bz * a.seg, z1 = min(z0 + a.seg, a.nz);
    const bool left = gx == 0;               // x = -1 is outside
    const bool right = gx + 4 >= a.nx;       // x = gx + 4 is outside
    const bool edge = bx == 0 || bx == a.ntx - 1;   // block-uniform
    const int cr = a.nx - 1 - gx;            // own cell of x = nx - 1 (right lanes)
    const int gxc = min(gx, (a.nx - 1) & ~3);   // lanes past the row's end read its last vector

    const int64_t plane = static_cast<int64_t>(a.pin) * a.ny;
    int off[VY], offu[R], offd[R];           // own rows, rows above and below (clamped)
#pragma unroll
    for (int v = 0; v < VY; ++v) off[v] = min(gy0 + v, a.ny - 1) * a.pin + gxc;
#pragma unroll
    for (int m = 0; m < R; ++m) {
        offu[m] = min(max(gy0 - 1 - m, 0), a.ny - 1) * a.pin + gxc;
        offd[m] = min(gy0 + VY + m, a.ny - 1) * a.pin + gxc;
    }
    const S *in = static_cast<const S *>(a.in);
    auto ok = [&](int64_t at, int n, int64_t limit) -> bool {
        if constexpr (CHK) {
            if (at >= 0 && at + n <= limit) return true;
            atomicOr(a.status, kStatusBounds);
            return false;
        } else {
            return true;
        }
    };
    // the last row ends with its cells, or with the pitch where vectors reach over them
    auto ok_in = [&](const S *p, int n) { return ok(p - in, n, plane * a.nz - (V ? 0 : a.pin - a.nx)); };
    auto load = [&](const S *p, float (&v)[4]) {   // p: cell gxc of a row
        if (!ok_in(p, V ? 4 : 1 + min(3, a.nx - 1 - gxc))) return;
        if constexpr (V) {
            Fmt<S>::load4(p, v);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = cell_in<S>(p + min(c, a.nx - 1 - gxc));
        }
    };
    auto zp = [&](int z) { return in + static_cast<int64_t>(min(max(z, 0), a.nz - 1)) * plane; };

    float q[Q][VY][4];
    grid_dep_wait();
#pragma unroll
    for (int j = 0; j < 2 * R + PF; ++j)
#pragma unroll
        for (int v = 0; v < VY; ++v) load(zp(z0 - R + j) + off[v], q[j][v]);

    S *const out = static_cast<S *>(a.out);
    for (int zb = z0; zb < z1; zb += Q) {
        SFor<0, Q>::run([&](auto Jc) {
            constexpr int J = decltype(Jc)::value;
            const int z = zb + J;
            if (z >= z1) return;
            {   // plane z + R + PF into the slot of plane z - R - 1
                const S *p = zp(z + R + PF);
#pragma unroll
                for (int v = 0; v < VY; ++v) load(p + off[v], q[(J + 2 * R + PF) % Q][v]);
            }
            auto qz = [&](int e) -> float (&)[VY][4] { return q[(J + R + e) % Q]; };   // plane z + e
            const S *pc = zp(z);
            float up[R][4], dn[R][4];
#pragma unroll
            for (int m = 0; m < R; ++m) {
                load(pc + offu[m], up[m]);
                load(pc + offd[m], dn[m]);
            }
            float(&ctr)[VY][4] = qz(0);
#pragma unroll
            for (int v = 0; v < VY; ++v) {
                float xl[R], xr[R];   // cells gx - 1 - k and gx + 4 + k
                if (edge && right) {  // cells past the row's end repeat its last cell
#pragma unroll
                    for (int c = 1; c < 4; ++c) ctr[v][c] = c > cr ? ctr[v][c - 1] : ctr[v][c];
                }
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    xl[k] = __shfl_up_sync(0xffffffffu, ctr[v][3 - k], 1, TX);
                    xr[k] = __shfl_down_sync(0xffffffffu, ctr[v][k], 1, TX);
                }
                if (tx == 0) {
                    float t[4];
                    if (left) {
                        t[0] = t[1] = t[2] = t[3] = ctr[v][0];
                    } else if constexpr (V) {
                        load(pc + off[v] - 4, t);
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (ok_in(pc + off[v] - 4 + c, 1)) t[c] = cell_in<S>(pc + off[v] - 4 + c);
                    }
#pragma unroll
                    for (int k = 0; k < R; ++k) xl[k] = t[3 - k];
                }
                if (tx == TX - 1 || (edge && right)) {
                    float t[4];
                    if (right) {
                        t[0] = t[1] = t[2] = t[3] = ctr[v][3];
                    } else if constexpr (V) {
                        load(pc + off[v] + 4, t);   // the row may end inside this vector
#pragma unroll
                        for (int c = 1; c < 4; ++c) t[c] = 4 + c > cr ? t[c - 1] : t[c];
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (ok_in(pc + off[v] + min(4 + c, cr), 1)) t[c] = cell_in<S>(pc + off[v] + min(4 + c, cr));
                    }
#pragma unroll
                    for (int k = 0; k < R; ++k) xr[k] = t[k];
                }
                auto xn = [&](int x) -> float { return x < 0 ? xl[cclamp(-x - 1, 0, R - 1)] : x > 3 ? xr[cclamp(x - 4, 0, R - 1)] : ctr[v][cclamp(x, 0, 3)]; };
                auto yn = [&](int y) -> const float * { return y < 0 ? up[cclamp(-y - 1, 0, R - 1)] : y >= VY ? dn[cclamp(y - VY, 0, R - 1)] : ctr[cclamp(y, 0, VY - 1)]; };
                float res[4];
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                    uint64_t acc = mul2(pk2(a.c[0], a.c[0]), pk2(ctr[v][c], ctr[v][c + 1]));
#pragma unroll
                    for (int i = 1; i <= R; ++i) {
                        const uint64_t so = pk2(yn(v - i)[c], yn(v - i)[c + 1]), no = pk2(yn(v + i)[c], yn(v + i)[c + 1]);
                        const uint64_t be = pk2(qz(-i)[v][c], qz(-i)[v][c + 1]), af = pk2(qz(i)[v][c], qz(i)[v][c + 1]);
                        if constexpr (SH) {
                            uint64_t sum;
                            if ((i & 1) == 0) sum = add2(pk2(xn(c - i), xn(c + 1 - i)), pk2(xn(c + i), xn(c + 1 + i)));
                            else sum = pk2(__fadd_rn(xn(c - i), xn(c + i)), __fadd_rn(xn(c + 1 - i), xn(c + 1 + i)));
                            sum = add2(add2(add2(add2(sum, so), no), be), af);
                            acc = fma2(pk2(a.c[i], a.c[i]), sum, acc);
                        } else {
                            const float *k = a.c + 6 * i - 5;
                            if ((i & 1) == 0) {
                                acc = fma2(pk2(k[0], k[0]), pk2(xn(c - i), xn(c + 1 - i)), acc);
                                acc = fma2(pk2(k[1], k[1]), pk2(xn(c + i), xn(c + 1 + i)), acc);
                            } else {
                                float a0, a1;
                                upk2(acc, a0, a1);
                                a0 = __fmaf_rn(k[0], xn(c - i), a0);
                                a1 = __fmaf_rn(k[0], xn(c + 1 - i), a1);
                                a0 = __fmaf_rn(k[1], xn(c + i), a0);
                                a1 = __fmaf_rn(k[1], xn(c + 1 + i), a1);
                                acc = pk2(a0, a1);
                            }
                            acc = fma2(pk2(k[2], k[2]), so, acc);
                            acc = fma2(pk2(k[3], k[3]), no, acc);
                            acc = fma2(pk2(k[4], k[4]), be, acc);
                            acc = fma2(pk2(k[5], k[5]), af, acc);
                        }
                    }
                    upk2(acc, res[c], res[c + 1]);
                }
                if (gx < a.nx && gy0 + v < a.ny) {
                    S *o = out + (static_cast<int64_t>(z) * a.ny + gy0 + v) * a.pout + gx;
                    if (!ok(o - out, a.vout ? 4 : min(4, a.nx - gx), static_cast<int64_t>(a.pout) * a.ny * a.nz)) continue;
                    if (a.vout) {
                        Fmt<S>::store4(o, res);
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (gx + c < a.nx) o[c] = to_storage<S>(res[c]);
                    }
                }
            }
        });
    }
}

}  // namespace stn
