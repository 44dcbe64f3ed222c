"""Batches of many grids of few kernel classes (persistent launches, also where 2D grids are far smaller than
the device) and of few grids per class (chains), against single runs, bit for bit."""
import pytest
import torch

import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import to_storage

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grids", [
    [(2, 1, (256, 256), 9, "f32")] * 40,
    [(2, 4, (128, 128), 7, "f32")] * 3 + [(3, 4, (40, 40, 40), 5, "f32")] * 3,
    [(3, 1 + k % 2, (16, 33, 32), 4 + k, "f32") for k in range(12)],
    [(3, r, (33, 32, 64), 7, "f32") for r in (1, 2, 3, 4) for _ in range(12)],
    [(2, 2, (200, 256), 10, "f32")] * 2 + [(3, 3, (20, 24, 40), 6, "bf16")] * 2])
def test_lists(grids):
    items, want, keep = [], [], []
    handles = {}
    for k, (dim, r, shape, iters, dt) in enumerate(grids):
        s = handles.setdefault((dim, r), st.Stencil(dim, r, gen.coefficients(dim, r)))
        x = to_storage(gen.uniform_grid(shape, seed=220 + k), dt).cuda()
        y = torch.full_like(x, float("nan"))
        nx, ny, nz = (shape[1], shape[0], 1) if dim == 2 else shape[::-1]
        items.append((s.handle, x.data_ptr(), y.data_ptr(), nx, ny, nz, iters, st.dtype_code(x)))
        want.append(s.run(x, iters))
        keep.append((x, y))
    for _ in range(2):
        for _, y in keep:
            y.fill_(float("nan"))
        st.stencil_run_batched(items, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert st.stencil_get_device_status() == 0
        for (_, y), w, g in zip(keep, want, grids):
            assert torch.equal(y, w), g
