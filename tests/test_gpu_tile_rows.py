"""Rows per thread of the library's rule in 3D: 4 where they gain more than their taller tiles round up."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import CODE, assert_bits_equal, oracle_passes, run_gpu, to_storage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,dt,ny,rows", [
    (2, "f16", 300, 2), (4, "bf16", 300, 2), (5, "f32", 300, 2), (2, "bf16", 512, 4), (4, "f16", 768, 4), (5, "f32", 512, 4),
    (3, "f16", 300, 4), (3, "f32", 300, 4), (4, "f32", 300, 4), (2, "f32", 512, 2), (6, "f32", 512, 2), (2, "f16", 40, 2),
    (2, "f16", 24, 4)])
def test_rule(r, dt, ny, rows):
    s = st.Stencil(3, r, gen.coefficients(3, r))
    assert s.default_schedule((100, ny, 1024), CODE[dt]).rows_per_thread == rows
    s.close()


@pytest.mark.parametrize("r,dt", [(2, "f16"), (5, "f32")])
@pytest.mark.parametrize("nx", [72, 73])
def test_bits_where_the_rows_change(r, dt, nx):
    c = gen.coefficients(3, r)
    s = st.Stencil(3, r, c)
    st.stencil_set_tile(s.handle, 1)   # padded copies for odd rows; marching passes off
    for ny in (31, 33, 48, 64):
        f = gen.uniform_grid((9, ny, nx), seed=230 + ny)
        x = to_storage(f, dt) if dt != "f32" else torch.from_numpy(f)
        want = oracle_passes(f, 3, r, c, 3, 1, dt) if dt != "f32" else oracle.sweep_f32(f, 3, r, c, 3)
        assert_bits_equal(run_gpu(s, x, 3), want, f"r={r} {dt} {nx}x{ny}")
    s.close()
