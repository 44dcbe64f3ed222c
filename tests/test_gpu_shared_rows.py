"""One coefficient per distance with two rows per step (2D streaming, radius 2 to 4), bit for bit
against its oracle: every compiled degree, odd and even segment starts, remainder passes, grids
narrower and shorter than a strip, and the rule's own choice."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import assert_bits_equal, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,t", [(2, 1), (2, 2), (2, 3), (3, 1), (3, 2), (4, 1), (4, 2)])
def test_shared_two_rows(r, t):
    c = gen.shared_coefficients(2, r)
    s = st.Stencil(2, r, c, shared=True)
    for ny, nx in ((203, 1000), (5, 8), (64, 516)):
        f = gen.uniform_grid((ny, nx), seed=110 + r)
        iters = 2 * t + 1
        want = oracle.sweep_shared_f32(f, 2, r, c, iters)
        for seg in (0, 1, 37):
            got = run_gpu(s, torch.from_numpy(f), iters, kernel=st.KERNEL_STREAM, t=t, planes_per_step=2, seg=seg)
            assert_bits_equal(got, want, f"shared r={r} t={t} {ny}x{nx} seg={seg}")
    s.close()


@pytest.mark.parametrize("r", [2, 3, 4])
def test_shared_rule_streams_two_rows(r):
    c = gen.shared_coefficients(2, r)
    s = st.Stencil(2, r, c, shared=True)
    st.stencil_set_tile(s.handle, -1)
    f = gen.uniform_grid((300, 1024), seed=120 + r)
    assert s.default_schedule(f.shape).planes_per_step == 2
    assert_bits_equal(run_gpu(s, torch.from_numpy(f), 5), oracle.sweep_shared_f32(f, 2, r, c, 5), f"shared rule r={r}")
    s.close()
