"""A warm-up with fewer steps than the captured run is enough: it leaves the scratch grid that the longer run needs
(more than one pass of the schedule), also where it ran as a single register-tile pass."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import assert_bits_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,r,shape,warm,iters,sched", [
    (2, 1, (256, 256), 10, 100, None), (2, 2, (200, 400), 4, 30, dict(t=3)), (2, 3, (90, 501), 2, 20, None),
    (3, 2, (20, 40, 64), 2, 9, None), (3, 1, (20, 40, 71), 2, 9, dict(kernel=st.KERNEL_NAIVE))])
def test_short_warm_up(dim, r, shape, warm, iters, sched):
    c = gen.coefficients(dim, r)
    s = st.Stencil(dim, r, c)
    other = st.Stencil(dim, r, c)
    sch = st.schedule(**sched) if sched else None
    f = gen.uniform_grid(shape, seed=250)
    x = torch.from_numpy(f).cuda()
    y = torch.empty_like(x)
    other.run(x, iters, out=y, sched=sch)   # loads the kernels
    s.run(x, warm, out=y)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        s.run(x, iters, out=y, sched=sch)
    y.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert_bits_equal(y.cpu(), oracle.sweep_f32(f, dim, r, c, iters), f"{dim}D r={r}")
    del g
    s.close()
