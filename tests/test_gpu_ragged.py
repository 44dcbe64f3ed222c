"""Grids whose rows are not whole 16-byte vectors, on streaming passes over a padded copy, bit for bit
against the oracle: rows ending on every cell of a vector and of a 64-cell tile, single rows and
planes, remainder passes, single passes, 16-bit storage (rounded at every step, like the one-step
kernel on such rows), buffers at any address, the allocation-free entry point and stream capture."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import assert_bits_equal, oracle_passes, to_storage

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (2, 3, 2), (5, 1, 3), (7, 17, 5), (19, 16, 62), (4, 33, 63), (9, 15, 65), (6, 20, 127), (3, 31, 130)]


def _run(s, x, iters):
    st.stencil_set_tile(s.handle, 1)
    out = s.run(x, iters)
    torch.cuda.synchronize()
    assert st.stencil_get_device_status() == 0
    return out.cpu()


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("r", [1, 2, 3, 4, 5, 6])
def test_fp32_rows_of_any_length(r, shared):
    c = gen.shared_coefficients(3, r) if shared else gen.coefficients(3, r)
    s = st.Stencil(3, r, c, shared=shared)
    for shape in SHAPES:
        f = gen.uniform_grid(shape, seed=80 + r)
        for iters in (1, 4, 5):
            want = (oracle.sweep_shared_f32 if shared else oracle.sweep_f32)(f, 3, r, c, iters)
            assert_bits_equal(_run(s, torch.from_numpy(f).cuda(), iters), want, f"r={r} {shape} iters={iters} shared={shared}")
    s.close()


@pytest.mark.parametrize("r", [2, 3, 4, 5])
def test_2d_rows_of_any_length(r):
    """2D streaming passes (strips of 512 columns less the halo) over a padded copy."""
    c = gen.coefficients(2, r)
    s = st.Stencil(2, r, c)
    st.stencil_set_tile(s.handle, 2)
    for shape in [(1, 1), (3, 2), (40, 7), (33, 497), (64, 510), (21, 1023), (130, 1025)]:
        f = gen.uniform_grid(shape, seed=85 + r)
        for iters in (1, 2, 7):
            want = oracle.sweep_f32(f, 2, r, c, iters)
            out = s.run(torch.from_numpy(f).cuda(), iters)
            torch.cuda.synchronize()
            assert st.stencil_get_device_status() == 0
            assert_bits_equal(out.cpu(), want, f"2D r={r} {shape} iters={iters}")
    s.close()


@pytest.mark.parametrize("dt", ["bf16", "f16"])
@pytest.mark.parametrize("r", [1, 2, 4, 6])
def test_16bit_rows_of_any_length(r, dt):
    c = gen.coefficients(3, r)
    s = st.Stencil(3, r, c)
    for shape in SHAPES + [(5, 9, 12), (5, 9, 68)]:   # 12 and 68 cells: whole 4-cell vectors, not 16 bytes
        f = gen.uniform_grid(shape, seed=90 + r)
        want = oracle_passes(f, 3, r, c, 3, 1, dt)
        assert_bits_equal(_run(s, to_storage(f, dt).cuda(), 3), want, f"{dt} r={r} {shape}")
    s.close()


def test_buffers_at_any_address_and_noalloc():
    r, shape, iters = 2, (12, 21, 99), 6
    n = 12 * 21 * 99
    c = gen.coefficients(3, r)
    s = st.Stencil(3, r, c)
    f = gen.uniform_grid(shape, seed=95)
    want = oracle.sweep_f32(f, 3, r, c, iters)
    for shift in (0, 1, 2, 3):
        a = torch.empty(n + 4, device="cuda")[shift:shift + n].view(shape)
        b = torch.full((n + 4,), float("nan"), device="cuda")
        a.copy_(torch.from_numpy(f))
        y = b[shift:shift + n].view(shape)
        for noalloc in (False, True):
            y.fill_(float("nan"))
            st.stencil_set_tile(s.handle, 1)
            if noalloc:
                st.stencil_run_noalloc(s.handle, a.data_ptr(), y.data_ptr(), 99, 21, 12, iters, 0,
                                       torch.cuda.current_stream().cuda_stream)
            else:
                s.run(a, iters, out=y)
            assert_bits_equal(y.cpu(), want, f"shift={shift} noalloc={noalloc}")
            assert torch.isnan(torch.cat([b[:shift], b[shift + n:]])).all()   # nothing else written
    s.close()


@pytest.mark.parametrize("dim,shape,r,iters", [(3, (12, 21, 99), 2, 1), (2, (200, 256), 4, 2)])
def test_capture_without_scratch_takes_the_route_that_needs_none(dim, shape, r, iters):
    """A first run under stream capture cannot allocate: calls whose streaming or one-step route needs
    no second grid are still captured, and replay to the same bits."""
    c = gen.coefficients(dim, r)
    f = gen.uniform_grid(shape, seed=96)
    x = torch.from_numpy(f).cuda()
    warm = st.Stencil(dim, r, c)
    st.stencil_set_tile(warm.handle, -1)
    warm.run(x, iters)                            # loads the kernels of that route
    s = st.Stencil(dim, r, c)
    if dim == 2:
        st.stencil_set_tile(s.handle, 1, 1, 8)    # two tile passes: they would need a second grid
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        s.run(x, iters, out=y)
    y.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert_bits_equal(y.cpu(), oracle.sweep_f32(f, dim, r, c, iters), f"{dim}D captured")
