"""2D streaming with two rows per step at radius 5 and 6 and four rows per step at radius 3, t = 2, bit for
bit against the oracle: segments starting on every row residue, grids shorter than the pipeline lag,
remainder passes, 16-bit storage, and the rule's own passes."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import assert_bits_equal, oracle_passes, run_gpu, to_storage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("r,t,p", [(5, 1, 2), (5, 2, 2), (6, 1, 2), (6, 2, 2), (3, 2, 4)])
def test_wide_rows(r, t, p, dt):
    if p == 4 and dt != "f32":
        pytest.skip("not compiled")
    c = gen.coefficients(2, r)
    s = st.Stencil(2, r, c)
    for ny, nx in ((203, 1008), (3, 8), (64, 520)):
        f = gen.uniform_grid((ny, nx), seed=160 + r)
        iters = 2 * t + 1
        want = oracle.sweep_f32(f, 2, r, c, iters) if dt == "f32" else oracle_passes(f, 2, r, c, iters, t, dt)
        x = torch.from_numpy(f) if dt == "f32" else to_storage(f, dt)
        assert st.stencil_resolve_schedule(s.handle, nx, ny, 1, st.dtype_code(x), st.schedule(
            kernel=st.KERNEL_STREAM, t=t, planes_per_step=p)).planes_per_step == p
        for seg in (0, 1, 6, 37):
            got = run_gpu(s, x, iters, kernel=st.KERNEL_STREAM, t=t, planes_per_step=p, seg=seg)
            assert_bits_equal(got, want, f"{dt} r={r} t={t} p={p} {ny}x{nx} seg={seg}")
    s.close()


@pytest.mark.parametrize("nx", [3000, 3001])
@pytest.mark.parametrize("r", [3, 5])
def test_rule_on_a_grid_that_streams(r, nx):
    """Few steps of a grid large enough for streaming passes (of a padded copy at 3001)."""
    c = gen.coefficients(2, r)
    s = st.Stencil(2, r, c)
    st.stencil_set_tile(s.handle, 2)
    f = gen.uniform_grid((700, nx), seed=170 + r)
    assert_bits_equal(run_gpu(s, torch.from_numpy(f), 5), oracle.sweep_f32(f, 2, r, c, 5), f"rule r={r} nx={nx}")
    s.close()
