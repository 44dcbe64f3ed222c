"""A schedule that names only the degree resolves to the pass that stencil_run_ex launches for it (2 rows per thread
in 3D), also where the rule's own passes have 4, which higher degrees are not compiled with."""
import pytest

import paper_2002_05983_gb300 as st
import stencil_inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,dt", [(3, st.STENCIL_BF16), (4, st.STENCIL_F16), (3, st.STENCIL_F32), (2, st.STENCIL_F16)])
@pytest.mark.parametrize("t", [1, 2])
def test_degree_alone(r, dt, t):
    s = st.Stencil(3, r, gen.coefficients(3, r))
    q = st.stencil_resolve_schedule(s.handle, 128, 128, 128, dt, st.schedule(t=t))
    assert (q.t, q.rows_per_thread) == (t, 2)
    f = list(st.stencil_schedule_features(s.handle, 128, 128, 128, dt, st.schedule(t=t)))
    assert f == list(st.stencil_schedule_features(s.handle, 128, 128, 128, dt, st.schedule(t=t, rows_per_thread=2)))
    s.close()
