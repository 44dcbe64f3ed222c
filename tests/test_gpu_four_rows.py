"""FP32 radius 3 on large 2D grids: four rows per step in the two-step passes alone; single steps (a call of one
step, the remainder of an odd number) keep two, which are faster there."""
import pytest
import torch

import paper_2002_05983_gb300 as st
import stencil_inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,iters,t,rows", [(8192, 1, 1, 2), (8192, 2, 2, 4), (8192, 7, 2, 4), (8184, 2, 2, 2)])
def test_rows_of_the_rule(n, iters, t, rows):
    s = st.Stencil(2, 3, gen.coefficients(2, 3))
    p = st.stencil_run_passes(s.handle, n, n, 1, iters, st.STENCIL_F32)
    assert (p.kind, p.t, p.planes_per_step) == (st.PASS_STREAM, t, rows)
    s.close()


def test_bits_of_a_remainder():
    s = st.Stencil(2, 3, gen.coefficients(2, 3))
    x = torch.rand((8192, 8192), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    y = s.run(x, 5)
    want = s.run(x, 5, sched=st.schedule(kernel=st.KERNEL_NAIVE))
    assert torch.equal(y, want)
    s.close()
