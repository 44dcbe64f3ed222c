"""Runs on rows of any length back to back on one stream, each reading what the run before it wrote: the
padded copy of a run is launched as a dependent of the last pass of the run before."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import assert_bits_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,r,shape,iters,mode", [
    (3, 1, (61, 70, 131), 4, 1), (3, 2, (40, 50, 67), 1, 1), (3, 4, (33, 40, 129), 2, 1), (2, 3, (700, 1021), 3, 2),
    (3, 2, (40, 50, 67), 3, 3), (2, 2, (300, 501), 5, 1)])
def test_runs_back_to_back(dim, r, shape, iters, mode):
    c = gen.coefficients(dim, r)
    s = st.Stencil(dim, r, c)
    st.stencil_set_tile(s.handle, mode)
    f = gen.uniform_grid(shape, seed=200 + r)
    x = torch.from_numpy(f).cuda()
    y = torch.empty_like(x)
    want = f
    for _ in range(3):
        s.run(x, iters, out=y)
        s.run(y, iters, out=x)
        want = oracle.sweep_f32(want, dim, r, c, 2 * iters)
    torch.cuda.synchronize()
    assert st.stencil_get_device_status() == 0
    assert_bits_equal(x.cpu(), want, f"{dim}D r={r} {shape}")
    s.close()
