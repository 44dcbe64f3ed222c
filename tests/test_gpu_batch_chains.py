"""Batched sweeps as one graph of per-grid chains and, for very long lists, as persistent launches:
both give stencil_run's bits (itself checked against the oracle elsewhere)."""
import pytest
import torch

import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import TORCH_DT, to_storage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grids", [
    # many 3D grids (more than the graph's branches), 16-bit storage, single passes and remainders
    [(3, 1 + k % 4, (5 + k, 9 + k, 8 * (1 + k % 5)), 1 + k % 7, ("f32", "bf16", "f16")[k % 3]) for k in range(19)]
    + [(2, 1 + k % 6, (40 + 7 * k, 8 * (3 + k)), 1 + 3 * k, ("f32", "bf16")[k % 2]) for k in range(7)],
    # 48 grids of three kernel classes: persistent launches
    [(2 + k % 2, 1 + k % 2, (9 + k, 40) if k % 2 == 0 else (5, 4 + k % 7, 24), 2 + k % 5, "f32") for k in range(48)],
    # 20001 passes of one grid: persistent launches
    [(3, 2, (4, 6, 8), 20001, "f32"), (2, 1, (20, 24), 11, "bf16")],
])
def test_batch_equals_single_runs(grids):
    items, want, keep = [], [], []
    for k, (dim, r, shape, iters, dt) in enumerate(grids):
        s = st.Stencil(dim, r, gen.coefficients(dim, r))
        x = to_storage(gen.workload_grid(dim, *shape[::-1], seed=70 + k), dt).cuda()
        y = torch.full_like(x, float("nan"))
        nx, ny, nz = (shape[1], shape[0], 1) if dim == 2 else shape[::-1]
        items.append((s.handle, x.data_ptr(), y.data_ptr(), nx, ny, nz, iters, st.dtype_code(x)))
        want.append(s.run(x, iters))
        assert want[-1].dtype == TORCH_DT[dt]
        keep.append((s, x, y))
    stream = torch.cuda.current_stream().cuda_stream
    for _ in range(2):   # the second call replays the cached graph
        for _, _, y in keep:
            y.fill_(float("nan"))
        st.stencil_run_batched(items, stream)
        torch.cuda.synchronize()
        assert st.stencil_get_device_status() == 0
        for (s, _, y), w, g in zip(keep, want, grids):
            assert torch.equal(y, w), g
