"""Register-tile passes of 2D grids, through the C ABI, bit for bit against the oracle.

Tiles are 128 columns wide (minus the halo) and 32 or 64 rows high; a lane owns 4 columns, a warp 4,
8 or 16 rows.  The grids end on and next to every one of those edges, the step counts split into
passes of unequal degree, and rows are of any length.  FP32: the same FMA chain as the oracle, so
equality is exact whatever the passes.  16-bit storage rounds after every step on rows that are not
whole 16-byte vectors and after every t steps of the default schedule otherwise, exactly like the
streaming and one-step kernels, whatever the passes."""
import numpy as np
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import CODE, assert_bits_equal, oracle_passes, to_storage

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (2, 3), (5, 2), (31, 4), (33, 127), (64, 128), (65, 129), (63, 120), (128, 113), (190, 260), (57, 501)]
TILES = [(4, 1), (4, 2), (8, 1), (8, 3), (16, 2), (16, 4)]   # rows per thread, most steps per pass


def _tiled(s, x, iters, t, rows):
    st.stencil_set_tile(s.handle, 1, t, rows)
    out = s.run(x, iters)
    torch.cuda.synchronize()
    assert st.stencil_get_device_status() == 0
    return out.cpu()


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("r", [1, 2, 3, 4, 5, 6])
def test_fp32_tiles_match_the_oracle(r, shared):
    iters = 7
    c = gen.shared_coefficients(2, r) if shared else gen.coefficients(2, r)
    s = st.Stencil(2, r, c, shared=shared)
    for ny, nx in SHAPES:
        f = gen.uniform_grid((ny, nx), seed=40 + r)
        want = (oracle.sweep_shared_f32 if shared else oracle.sweep_f32)(f, 2, r, c, iters)
        x = torch.from_numpy(f).cuda()
        for rows, t in TILES:
            if r > 4 and rows == 4 or 8 * r * t > 3 * (32 if rows == 4 else 64):
                continue   # not compiled, or the halo leaves too little of a tile
            assert_bits_equal(_tiled(s, x, iters, t, rows), want, f"r={r} {ny}x{nx} rows={rows} t={t} shared={shared}")
    s.close()


@pytest.mark.parametrize("dt", ["bf16", "f16"])
@pytest.mark.parametrize("r", [1, 3, 4, 6])
def test_16bit_tiles_round_where_the_rule_does(r, dt):
    c = gen.coefficients(2, r)
    s = st.Stencil(2, r, c)
    for ny, nx in ((65, 136), (70, 129), (40, 260), (33, 12)):
        f = gen.uniform_grid((ny, nx), seed=50 + r)
        x = to_storage(f, dt).cuda()
        t = s.default_schedule((ny, nx), CODE[dt]).t if nx % 8 == 0 else 1
        iters = 3 * t + 1
        want = oracle_passes(f, 2, r, c, iters, t, dt)
        for most in {t, 2 * t}:
            for rows in (8, 16):
                if 8 * r * most <= 3 * 64:
                    assert_bits_equal(_tiled(s, x, iters, most, rows), want, f"{dt} r={r} {ny}x{nx} rows={rows} t={most}")
    s.close()


def test_unaligned_buffers_and_the_rule_itself():
    """Grids at addresses that are not multiples of 16 bytes (rows of any length), the rule's own
    choice of kernel, and the allocation-free entry point."""
    for r, ny, nx, iters in ((1, 200, 333, 23), (4, 90, 515, 9), (2, 300, 1024, 40), (3, 1000, 7, 5)):
        c = gen.coefficients(2, r)
        s = st.Stencil(2, r, c)
        f = gen.uniform_grid((ny, nx), seed=60)
        want = oracle.sweep_f32(f, 2, r, c, iters)
        for shift in ((0,) if nx % 4 == 0 else (0, 1, 3)):
            a = torch.empty(ny * nx + 4, device="cuda")[shift:shift + ny * nx].view(ny, nx)
            b = torch.full((ny * nx + 4,), float("nan"), device="cuda")
            a.copy_(torch.from_numpy(f))
            y = b[shift:shift + ny * nx].view(ny, nx)
            s.run(a, iters, out=y)
            assert_bits_equal(y.cpu(), want, f"r={r} {ny}x{nx} shift={shift}")
            rest = torch.cat([b[:shift], b[shift + ny * nx:]])
            assert torch.isnan(rest).all()   # nothing outside the grid was written
            y.fill_(float("nan"))
            st.stencil_run_noalloc(s.handle, a.data_ptr(), y.data_ptr(), nx, ny, 1, iters, 0,
                                   torch.cuda.current_stream().cuda_stream)
            assert_bits_equal(y.cpu(), want, f"noalloc r={r} {ny}x{nx} shift={shift}")
        s.close()


@pytest.mark.parametrize("dt", ["f32", "bf16", "f16"])
def test_special_values_through_tiles(dt):
    """Infinities, NaN, signed zeros, subnormals and the largest finite values."""
    r, ny, nx, iters = 2, 70, 133, 3
    f = gen.uniform_grid((ny, nx), seed=61)
    big = {"f32": 3.4028235e38, "bf16": 3.3895e38, "f16": 65504.0}[dt]
    f.reshape(-1)[::97] = np.resize(np.array([np.inf, -np.inf, np.nan, -0.0, 0.0, 1e-42, big, -big], np.float32),
                                    f.reshape(-1)[::97].shape)
    c = gen.coefficients(2, r)
    s = st.Stencil(2, r, c)
    x = to_storage(f, dt).cuda() if dt != "f32" else torch.from_numpy(f).cuda()
    with np.errstate(all="ignore"):
        want = oracle.sweep_f32(f, 2, r, c, iters) if dt == "f32" else oracle_passes(f, 2, r, c, iters, 1, dt)
    got = _tiled(s, x, iters, 2, 8).float().numpy()
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint32), want[~nan].astype(np.float32).view(np.uint32))
    s.close()
