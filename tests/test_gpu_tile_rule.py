"""Register tiles or streaming passes: problems on which the estimates are close and tiles measured slower stream."""
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
