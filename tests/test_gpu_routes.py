"""The kernels the library's rule picks (stencil_run_passes), and every one of them under stream capture:
a warmed-up run is captured with its dependent launches and replays on new data to the oracle's bits."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import assert_bits_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,r,shape,iters,kind", [
    (2, 1, (256, 256), 10, st.PASS_TILE), (2, 1, (16384, 16384), 1000, st.PASS_TILE),
    (2, 4, (16384, 16384), 1000, st.PASS_STREAM), (2, 3, (2047, 3001), 50, st.PASS_TILE),
    (2, 4, (16383, 16381), 50, st.PASS_PADDED), (3, 2, (96, 96, 96), 100, st.PASS_MARCH),
    (3, 4, (512, 512, 512), 50, st.PASS_STREAM), (3, 1, (237, 243, 251), 50, st.PASS_PADDED)])
def test_rule_picks(dim, r, shape, iters, kind):
    s = st.Stencil(dim, r, gen.coefficients(dim, r))
    nx, ny, nz = (shape[1], shape[0], 1) if dim == 2 else shape[::-1]
    p = st.stencil_run_passes(s.handle, nx, ny, nz, iters, st.STENCIL_F32)
    assert p.kind == kind and 1 <= p.t <= iters
    passes = p.launches - (1 if kind == st.PASS_PADDED else 0)
    assert passes * p.t >= iters > (passes - 1)
    st.stencil_set_tile(s.handle, -1)
    q = st.stencil_run_passes(s.handle, nx, ny, nz, iters, st.STENCIL_F32)
    assert q.kind == (st.PASS_STREAM if nx % 4 == 0 else st.PASS_NAIVE)
    s.close()


@pytest.mark.parametrize("dim,r,shape,iters,mode", [
    (2, 2, (300, 400), 23, 1), (2, 3, (90, 501), 12, 1), (2, 4, (90, 501), 5, 2), (3, 2, (20, 40, 64), 7, 3),
    (3, 3, (20, 40, 71), 5, 3), (3, 2, (20, 40, 71), 6, 1), (3, 4, (30, 40, 64), 4, -1), (3, 1, (30, 40, 64), 5, -1)])
def test_every_route_under_capture(dim, r, shape, iters, mode):
    c = gen.coefficients(dim, r)
    s = st.Stencil(dim, r, c)
    st.stencil_set_tile(s.handle, mode)
    x = torch.empty(shape, device="cuda").zero_()
    y = torch.empty_like(x)
    s.run(x, iters, out=y)   # allocates the scratch grids and loads the kernels
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        s.run(x, iters, out=y)
    for seed in (180, 181):
        f = gen.uniform_grid(shape, seed=seed)
        x.copy_(torch.from_numpy(f))
        y.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert_bits_equal(y.cpu(), oracle.sweep_f32(f, dim, r, c, iters), f"{dim}D r={r} mode={mode} seed={seed}")
    assert st.stencil_get_device_status() == 0
    del g
    s.close()
