"""Automatic segment lengths of 3D streaming passes: whole waves for the library's own degree and rows per
thread and where a schedule leaves most of the device empty, four waves of at least 64 planes for the other
schedules (whole waves made some of them up to 24 % slower) and for radius 1 from one wave on (up to 8 %)."""
import pytest

import paper_2002_05983_gb300 as st
import stencil_inputs as gen

pytestmark = pytest.mark.gpu


def _seg(r, dt, n, **sched):
    s = st.Stencil(3, r, gen.coefficients(3, r))
    seg = st.stencil_resolve_schedule(s.handle, *n, dt, st.schedule(**sched)).seg
    s.close()
    return seg


@pytest.mark.parametrize("r,dt,n,sched,seg", [
    (2, st.STENCIL_F32, (512, 512, 512), dict(t=1, rows_per_thread=4), 64),
    (2, st.STENCIL_F32, (384, 384, 384), dict(t=1, rows_per_thread=4), 64),
    (1, st.STENCIL_F32, (1024, 300, 100), dict(t=3, rows_per_thread=2), 72),
    (3, st.STENCIL_F32, (256, 256, 256), dict(t=2, rows_per_thread=2), 112),
    (2, st.STENCIL_F16, (1024, 300, 100), dict(t=2, rows_per_thread=2), 80),
    (1, st.STENCIL_F32, (368, 653, 154), dict(), 64), (1, st.STENCIL_F32, (400, 400, 400), dict(), 64),
    (1, st.STENCIL_F16, (1024, 300, 100), dict(), 64)])
def test_other_schedules_keep_four_waves(r, dt, n, sched, seg):
    assert _seg(r, dt, n, **sched) == seg


@pytest.mark.parametrize("r,n,sched", [
    (3, (512, 512, 512), dict()), (3, (512, 512, 512), dict(t=1, rows_per_thread=4)), (1, (256, 256, 256), dict()),
    (2, (96, 96, 96), dict(t=1, rows_per_thread=4)), (1, (96, 96, 96), dict(t=3, rows_per_thread=2))])
def test_whole_waves(r, n, sched):
    assert _seg(r, st.STENCIL_F32, n, **sched) not in (64, 72, 96)
