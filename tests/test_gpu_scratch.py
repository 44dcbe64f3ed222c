"""A graph captured from a run keeps working after the same handle has run larger problems and problems on other
kernels, which need a larger scratch buffer."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import assert_bits_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,r,shape,iters,sched", [
    (3, 1, (30, 40, 71), 6, None), (2, 3, (90, 501), 40, None), (3, 2, (30, 40, 64), 4, dict(t=1)), (2, 2, (90, 512), 40, None),
    (3, 4, (20, 40, 71), 3, dict(kernel=st.KERNEL_NAIVE))])
def test_graph_replays_after_growth(dim, r, shape, iters, sched):
    c = gen.coefficients(dim, r)
    s = st.Stencil(dim, r, c)
    sch = st.schedule(**sched) if sched else None
    x = torch.zeros(shape, device="cuda")
    y = torch.empty_like(x)
    s.run(x, iters, out=y, sched=sch)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        s.run(x, iters, out=y, sched=sch)
    hold = []
    for grow in (shape, tuple(2 * n + 1 for n in shape), tuple(3 * n for n in shape)):
        z = torch.ones(grow, device="cuda")
        s.run(z, iters)
        s.run(z, iters, sched=st.schedule(kernel=st.KERNEL_NAIVE))
        hold.append(torch.full((256 * 1024,), float("nan"), device="cuda"))   # memory that a freed buffer left
    f = gen.uniform_grid(shape, seed=240)
    x.copy_(torch.from_numpy(f))
    y.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert_bits_equal(y.cpu(), oracle.sweep_f32(f, dim, r, c, iters), f"{dim}D r={r}")
    del g
    s.close()
