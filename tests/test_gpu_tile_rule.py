"""Register tiles or streaming passes, padded copies or the one-step kernel: problems on which the estimates are close
take the kernel that measured faster."""
import pytest

import paper_2002_05983_gb300 as st
import stencil_inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,dt,shape,iters,kind", [
    (3, st.STENCIL_F32, (4096, 4096), 1, st.PASS_STREAM), (3, st.STENCIL_F32, (1024, 16384), 1, st.PASS_STREAM),
    (3, st.STENCIL_F32, (16384, 1024), 1, st.PASS_STREAM), (4, st.STENCIL_F32, (4096, 4096), 7, st.PASS_STREAM),
    (6, st.STENCIL_F32, (12000, 12000), 1, st.PASS_STREAM), (6, st.STENCIL_F16, (12000, 12000), 1, st.PASS_STREAM),
    (5, st.STENCIL_F32, (9955, 3832), 3, st.PASS_STREAM), (1, st.STENCIL_F32, (16384, 16384), 1000, st.PASS_TILE),
    (2, st.STENCIL_F32, (4096, 4096), 100, st.PASS_TILE), (4, st.STENCIL_F32, (4096, 4096), 100, st.PASS_TILE),
    (6, st.STENCIL_F32, (4096, 4096), 1, st.PASS_TILE), (1, st.STENCIL_F32, (256, 256), 10, st.PASS_TILE)])
def test_close_calls(r, dt, shape, iters, kind):
    s = st.Stencil(2, r, gen.coefficients(2, r))
    assert st.stencil_run_passes(s.handle, shape[1], shape[0], 1, iters, dt).kind == kind
    s.close()


@pytest.mark.parametrize("r,dt,shape,iters,shared,kind", [
    (1, st.STENCIL_F16, (530, 651, 25), 1, False, st.PASS_NAIVE), (1, st.STENCIL_F32, (168, 513, 18), 2, True, st.PASS_NAIVE),
    (1, st.STENCIL_F32, (237, 243, 251), 50, False, st.PASS_PADDED), (1, st.STENCIL_F32, (237, 243, 251), 2, False, st.PASS_PADDED),
    (4, st.STENCIL_F16, (200, 300, 333), 2, False, st.PASS_PADDED)])
def test_padded_or_one_step(r, dt, shape, iters, shared, kind):
    s = st.Stencil(3, r, gen.shared_coefficients(3, r) if shared else gen.coefficients(3, r), shared=shared)
    assert st.stencil_run_passes(s.handle, *shape[::-1], iters, dt).kind == kind
    s.close()
