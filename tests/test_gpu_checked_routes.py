"""Bounds-checked instantiations of the rule's other kernels: register tiles, marching passes and streaming passes
over padded rows, on grids whose ends fall everywhere in vectors and tiles, report no access out of range and
match the oracle."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import CODE, assert_bits_equal, oracle_passes, to_storage

pytestmark = pytest.mark.gpu

SHAPES2 = [(1, 1), (3, 2), (33, 127), (65, 129), (40, 7), (21, 511), (130, 517)]
SHAPES3 = [(1, 1, 1), (2, 3, 2), (7, 17, 5), (19, 16, 62), (4, 33, 63), (9, 15, 65), (6, 20, 127), (3, 31, 130)]


@pytest.mark.parametrize("dim,r,dt,shared,mode,rows,t,kind", [
    (2, 1, "f32", False, 1, 4, 3, st.PASS_TILE), (2, 3, "f32", False, 1, 8, 2, st.PASS_TILE),
    (2, 6, "f32", False, 1, 8, 1, st.PASS_TILE), (2, 4, "bf16", False, 1, 16, 2, st.PASS_TILE),
    (2, 2, "f32", True, 1, 16, 4, st.PASS_TILE), (2, 4, "f32", False, 2, 0, 0, st.PASS_PADDED),
    (3, 1, "f32", False, 3, 0, 0, st.PASS_MARCH), (3, 4, "f32", False, 3, 0, 0, st.PASS_MARCH),
    (3, 3, "f16", False, 3, 0, 0, st.PASS_MARCH), (3, 2, "f32", True, 3, 0, 0, st.PASS_MARCH),
    (3, 1, "f32", False, 1, 0, 0, st.PASS_PADDED), (3, 4, "f32", False, 1, 0, 0, st.PASS_PADDED),
    (3, 2, "f16", False, 1, 0, 0, st.PASS_PADDED)])
def test_no_access_out_of_range(dim, r, dt, shared, mode, rows, t, kind):
    c = gen.shared_coefficients(dim, r) if shared else gen.coefficients(dim, r)
    s = st.Stencil(dim, r, c, shared=shared)
    st.stencil_set_checked(s.handle, True)
    st.stencil_set_tile(s.handle, mode, t, rows)
    assert st.stencil_get_device_status(clear=True) == 0
    for shape in SHAPES2 if dim == 2 else SHAPES3:
        f = gen.uniform_grid(shape, seed=270 + r)
        nx, ny, nz = (shape[1], shape[0], 1) if dim == 2 else shape[::-1]
        x = torch.from_numpy(f).cuda() if dt == "f32" else to_storage(f, dt).cuda()
        for iters in (1, 5):
            p = st.stencil_run_passes(s.handle, nx, ny, nz, iters, CODE[dt])
            assert p.kind == kind and (not rows or p.rows_per_thread == rows), (shape, p.kind)
            got = s.run(x, iters)
            torch.cuda.synchronize()
            assert st.stencil_get_device_status(clear=True) == 0, (shape, iters)
            want = ((oracle.sweep_shared_f32 if shared else oracle.sweep_f32)(f, dim, r, c, iters) if dt == "f32"
                    else oracle_passes(f, dim, r, c, iters, 1, dt))
            assert_bits_equal(got.cpu(), want, f"{shape} iters={iters}")
    s.close()
