"""The kernels that stencil_set_tile asks for are the ones that run (stencil_run_passes), in as many launches as their
degree needs, and infinities, NaN, signed zeros, subnormals and the largest finite values go through marching passes
and padded rows as through the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import CODE, oracle_passes, to_storage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,r,dt,shape,iters,mode,t,rows,kind,launches", [
    (2, 1, "f32", (65, 129), 7, 1, 3, 8, st.PASS_TILE, 3), (2, 1, "f32", (65, 129), 7, 1, 2, 4, st.PASS_TILE, 4),
    (2, 4, "f32", (63, 120), 7, 1, 2, 16, st.PASS_TILE, 4), (2, 6, "f32", (190, 260), 7, 1, 1, 8, st.PASS_TILE, 7),
    (2, 3, "bf16", (65, 136), 10, 1, 3, 16, st.PASS_TILE, 4), (2, 3, "bf16", (70, 129), 4, 1, 1, 8, st.PASS_TILE, 4),
    (2, 4, "f16", (65, 136), 7, 1, 4, 16, st.PASS_TILE, 2),
    (2, 2, "f32", (40, 7), 7, 2, 0, 0, st.PASS_PADDED, 4), (2, 3, "f32", (33, 497), 7, 2, 0, 0, st.PASS_PADDED, 5),
    (2, 5, "f32", (130, 1025), 2, 2, 0, 0, st.PASS_PADDED, 2), (2, 3, "f32", (700, 3000), 5, 2, 0, 0, st.PASS_STREAM, 3),
    (3, 1, "f32", (9, 15, 65), 5, 1, 0, 0, st.PASS_PADDED, 4), (3, 4, "f32", (4, 33, 63), 4, 1, 0, 0, st.PASS_PADDED, 5),
    (3, 1, "bf16", (9, 15, 65), 3, 1, 0, 0, st.PASS_PADDED, 4), (3, 2, "f16", (5, 9, 68), 3, 1, 0, 0, st.PASS_PADDED, 4),
    (3, 1, "f32", (20, 16, 64), 5, 3, 0, 0, st.PASS_MARCH, 5), (3, 4, "f16", (6, 17, 68), 3, 3, 0, 0, st.PASS_MARCH, 3),
    (3, 3, "f32", (9, 17, 65), 2, 3, 0, 0, st.PASS_MARCH, 2)])
def test_the_kernel_asked_for(dim, r, dt, shape, iters, mode, t, rows, kind, launches):
    s = st.Stencil(dim, r, gen.coefficients(dim, r))
    st.stencil_set_tile(s.handle, mode, t, rows)
    nx, ny, nz = (shape[1], shape[0], 1) if dim == 2 else shape[::-1]
    p = st.stencil_run_passes(s.handle, nx, ny, nz, iters, CODE[dt])
    assert (p.kind, p.launches) == (kind, launches)
    if kind == st.PASS_TILE:
        assert p.rows_per_thread == rows and p.t <= t
    s.close()


@pytest.mark.parametrize("dim,r,shape,mode,kind,dt", [(3, *p, dt) for dt in ("f32", "bf16", "f16") for p in (
    (2, (9, 18, 67), 3, st.PASS_MARCH), (4, (7, 33, 130), 3, st.PASS_MARCH), (2, (9, 18, 64), 3, st.PASS_MARCH),
    (1, (9, 18, 67), 1, st.PASS_PADDED), (4, (7, 33, 130), 1, st.PASS_PADDED))] + [(2, 4, (40, 517), 2, st.PASS_PADDED, "f32")])
def test_special_values(dim, r, shape, mode, kind, dt):
    iters = 3
    f = gen.uniform_grid(shape, seed=280 + r)
    big = {"f32": 3.4028235e38, "bf16": 3.3895e38, "f16": 65504.0}[dt]
    special = np.array([np.inf, -np.inf, np.nan, -0.0, 0.0, 1e-42, big, -big], np.float32)
    flat = f.reshape(-1)
    flat[::997] = np.resize(special, flat[::997].shape)
    f[..., -1].reshape(-1)[::53] = np.resize(special[3:], f[..., -1].reshape(-1)[::53].shape)   # at rows' ends too
    c = gen.coefficients(dim, r)
    s = st.Stencil(dim, r, c)
    st.stencil_set_tile(s.handle, mode)
    x = to_storage(f, dt).cuda() if dt != "f32" else torch.from_numpy(f).cuda()
    nx, ny, nz = (shape[1], shape[0], 1) if dim == 2 else shape[::-1]
    assert st.stencil_run_passes(s.handle, nx, ny, nz, iters, CODE[dt]).kind == kind
    with np.errstate(all="ignore"):
        want = oracle.sweep_f32(f, dim, r, c, iters) if dt == "f32" else oracle_passes(f, dim, r, c, iters, 1, dt)
    got = s.run(x, iters).cpu().float().numpy()
    nan = np.isnan(want)
    assert nan.any() and not nan.all()
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint32), want[~nan].astype(np.float32).view(np.uint32))
    s.close()
