"""The sweeps that users of the package run, as measurable cases.

A case is one call of the public API on grids that already sit in device memory, with the
handle, the input and the output buffer a program keeps between calls:

  kind "sweep": ``Stencil.run`` with the library's own schedule: 2D or 3D, radius 1..6, FP32,
                BF16 or FP16 storage, one coefficient per (distance, direction) or one per
                distance, any size (rows of any length, not only whole 16-byte vectors);
  kind "batch": ``stencil_run_batched`` over a list of mixed grids (2D and 3D, FP32 and BF16,
                radius 1..4) described by the numbers ``n2``, ``n3`` and ``mix``.

Sizes: the benchmark's workloads (16384^2, 512^3, 768^3 in 16 bits, 256^2 for 10 steps, batches
of sides 512..8192 and 64..384) and generic ones between them.
"""
import math
import random

import numpy as np
import torch

import paper_2002_05983_gb300 as st

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _sweep(nx, ny, nz, radius, iters, dtype="f32", shared=False):
    return {"kind": "sweep", "nx": nx, "ny": ny, "nz": nz, "radius": radius, "iters": iters, "dtype": dtype,
            "shared": shared}


def listed():
    return [
        # a first try, or one call inside a larger program: launches and latency are everything
        {"name": "tiny_2d_r1"} | _sweep(256, 256, 0, 1, 10),
        # an ordinary image-sized field, relaxed for a while
        {"name": "small_2d_r2"} | _sweep(1024, 1024, 0, 2, 100),
        # the paper's 2D workload at its largest radius
        {"name": "large_2d_r4"} | _sweep(16384, 16384, 0, 4, 100),
        # a field with its boundary points counted: rows that are not whole 16-byte vectors
        {"name": "odd_2d_r3"} | _sweep(3001, 2047, 0, 3, 50),
        # 2D precision workload: half the bytes per cell
        {"name": "half_2d_r4"} | _sweep(16384, 16384, 0, 4, 100, "bf16"),
        # one coefficient per distance, the form of the codes the paper compares with
        {"name": "shared_2d_r2"} | _sweep(8192, 8192, 0, 2, 60, "f32", True),
        # a small 3D block, as one part of a decomposed domain
        {"name": "small_3d_r2"} | _sweep(96, 96, 96, 2, 100),
        # the paper's 3D workload at its smallest and its largest radius
        {"name": "large_3d_r1"} | _sweep(512, 512, 512, 1, 50),
        {"name": "large_3d_r4"} | _sweep(512, 512, 512, 4, 50),
        # 3D precision workload
        {"name": "half_3d_r4"} | _sweep(768, 768, 768, 4, 20, "f16"),
        # a 3D field with odd extents
        {"name": "odd_3d_r1"} | _sweep(251, 243, 237, 1, 50),
        # a serving-style batch of mixed grids
        {"name": "batch_mixed", "kind": "batch", "n2": 16, "n3": 8, "mix": 2, "iters": 100},
    ]


# the most a drawn case may cost, in FLOP (below the largest listed one)
_MOST_FLOPS = 16384 * 16384 * 100 * 33


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: sizes spread over their logarithm, a quarter of the
    sweeps with rows of any length, the rest in rows of 8 cells times a whole number."""
    if rng.random() < 0.1:
        case = {"kind": "batch", "n2": rng.randint(2, 16), "n3": rng.randint(1, 8), "mix": rng.randint(3, 1 << 20),
                "iters": 1}
        return case | {"iters": min(rng.randint(20, 99), _MOST_FLOPS // work(case)["flops"])}
    dim = rng.choice([2, 3])
    radius = rng.randint(5, 6) if rng.random() < 0.08 else rng.randint(1, 4)
    shared = rng.random() < 0.12
    dtype = "f32" if shared or rng.random() < 0.6 else rng.choice(["bf16", "f16"])
    lo, hi = (256, 16384) if dim == 2 else (64, 768)
    nx, ny, nz = (_log_int(rng, lo, hi) for _ in range(3))
    nz = nz if dim == 3 else 0
    if rng.random() < 0.75:
        nx = max(8, nx // 8 * 8)
    flops = 2 * (2 * dim * radius) + 1
    cells = nx * ny * max(nz, 1)
    most = max(1, min(100, _MOST_FLOPS // (cells * flops)))
    iters = _log_int(rng, min(10, most), most)
    return _sweep(nx, ny, nz, radius, iters, dtype, shared)


def _grids(case):
    """The grids of a case: dicts of sizes, radius, dtype and coefficient form."""
    if case["kind"] == "sweep":
        return [{k: case[k] for k in ("nx", "ny", "nz", "radius", "dtype", "shared")}]
    rng = random.Random(1000003 * case["mix"] + 17)
    out = []
    for i in range(case["n2"] + case["n3"]):
        two = i < case["n2"]
        lo, hi = (512, 8192) if two else (64, 384)
        nx, ny, nz = (rng.randint(lo, hi) for _ in range(3))
        out.append({"nx": nx // 8 * 8, "ny": ny, "nz": 0 if two else nz, "radius": rng.randint(1, 4),
                    "dtype": rng.choice(["f32", "bf16"]), "shared": False})
    return out


def _coefficients(g, rng):
    """Nonnegative weights whose operator row sums to about 1, as FP32."""
    dim = 3 if g["nz"] else 2
    k = 1 + g["radius"] * (1 if g["shared"] else 2 * dim)
    w = rng.random(k) + 2.0 ** -25
    total = w[0] + 2 * dim * w[1:].sum() if g["shared"] else w.sum()
    return (w / total).astype(np.float32)


def _inputs(case, seed):
    """[(grid, coefficients, field)]: uniform [0, 1) values, in 3D with a Gaussian bump of sigma
    16 cells at the centre, rounded to the storage type."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for g in _grids(case):
        dim = 3 if g["nz"] else 2
        shape = (g["nz"], g["ny"], g["nx"]) if dim == 3 else (g["ny"], g["nx"])
        f = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32)
        if dim == 3:
            e = [torch.exp(-(torch.arange(n, device="cuda", dtype=torch.float32) - n // 2) ** 2 / 512.0) for n in shape]
            f.addcmul_((e[0][:, None] * e[1][None, :])[:, :, None], e[2][None, None, :])
        out.append((g, _coefficients(g, rng), f.to(DTYPES[g["dtype"]])))
    return out


def prepare(case, seed):
    grids = []
    for g, c, x in _inputs(case, seed):
        s = st.Stencil(3 if g["nz"] else 2, g["radius"], c, shared=g["shared"])
        grids.append((s, x, torch.empty_like(x)))
    state = {"iters": case["iters"], "grids": grids}
    if case["kind"] == "batch":
        state["items"] = [st.BatchItem(s.handle, x.data_ptr(), y.data_ptr(), g["nx"], g["ny"], max(g["nz"], 1),
                                       case["iters"], st.dtype_code(x))
                          for g, (s, x, y) in zip(_grids(case), grids)]
    return state


def run(state):
    if "items" in state:
        st.stencil_run_batched(state["items"], torch.cuda.current_stream().cuda_stream)
        return [y for _, _, y in state["grids"]]
    s, x, y = state["grids"][0]
    return s.run(x, state["iters"], out=y)


def work(case):
    """Each input cell read once, each output cell written once; 1 multiply and one multiply-add
    per neighbour and cell update (shared coefficients: 2D adds and one more operation per distance)."""
    nbytes = flops = 0
    for g in _grids(case):
        dim = 3 if g["nz"] else 2
        cells = g["nx"] * g["ny"] * max(g["nz"], 1)
        nbytes += 2 * cells * (4 if g["dtype"] == "f32" else 2)
        per_cell = 1 + g["radius"] * ((2 * dim + 1) if g["shared"] else 4 * dim)
        flops += cells * case["iters"] * per_cell
    return {"bytes": nbytes, "flops": flops}


def _sweep64(f, g, c, iters):
    """The definition in FP64: every neighbour outside the grid is the border cell."""
    r, axes = g["radius"], list(range(f.dim() - 1, -1, -1))   # x, y[, z]
    n = f.shape
    acc = f.double()
    p = torch.empty([k + 2 * r for k in n], device=f.device, dtype=torch.float64)
    mid = tuple(slice(r, r + k) for k in n)
    c = [float(v) for v in c]

    def near(axis, step):
        return p[tuple(slice(r + step, r + step + n[a]) if a == axis else mid[a] for a in range(len(n)))]

    for _ in range(iters):
        p[mid] = acc
        for a in axes:   # the star reads only the sides of the frame, not its corners
            for lo, hi, src in ((0, r, r), (r + n[a], 2 * r + n[a], r + n[a] - 1)):
                at = [mid[b] for b in range(len(n))]
                at[a] = slice(src, src + 1)
                to = list(at)
                to[a] = slice(lo, hi)
                p[tuple(to)] = p[tuple(at)]
        torch.mul(p[mid], c[0], out=acc)
        for i in range(1, r + 1):
            for d, (a, sign) in enumerate((a, sign) for a in axes for sign in (-1, 1)):
                acc.add_(near(a, sign * i), alpha=c[i] if g["shared"] else c[1 + (i - 1) * 2 * len(n) + d])
    return acc


def exact(case, seed):
    # FP64 sweeps cost about a dozen passes over FP64 grids per step
    if sum(g["nx"] * g["ny"] * max(g["nz"], 1) * (1 + 2 * g["radius"] * (3 if g["nz"] else 2)) for g in _grids(case)) \
            * case["iters"] > 1.5e12:
        return None
    outs = [_sweep64(f, g, c, case["iters"]) for g, c, f in _inputs(case, seed)]
    return outs if case["kind"] == "batch" else outs[0]
