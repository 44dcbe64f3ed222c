"""Schedules that name the prefetch depth of a kernel's earlier form keep running: picks kept in a tuning-cache
file and explicit schedules.  3D one-level kernels of radius 4 to 6, and of radius 2 with 16-bit storage and 4
rows per thread, loaded 2 planes ahead before they took two steps per chunk; 2D radius 5 and 6 and the shared
form had one row per step (5, 6 and, at radius 2 and t = 3, 7 rows ahead), radius 3 at t = 2 two (10 ahead)."""
import pytest
import torch

import oracle
import paper_2002_05983_gb300 as st
import stencil_inputs as gen
from gpu_util import CODE, assert_bits_equal, oracle_passes, to_storage

pytestmark = pytest.mark.gpu


def _problem(dim, r, dt, shape, t, iters, shared=False):
    c = gen.shared_coefficients(dim, r) if shared else gen.coefficients(dim, r)
    f = gen.uniform_grid(shape, seed=210 + r)
    if dt == "f32":
        want = (oracle.sweep_shared_f32 if shared else oracle.sweep_f32)(f, dim, r, c, iters)
        return c, torch.from_numpy(f).cuda(), want
    return c, to_storage(f, dt).cuda(), oracle_passes(f, dim, r, c, iters, t, dt)


@pytest.mark.parametrize("version", ["v1", "v2"])
@pytest.mark.parametrize("r,dt,rows", [(4, "f32", 4), (4, "f32", 2), (5, "f32", 2), (6, "f32", 2), (4, "bf16", 2), (2, "f16", 4)])
def test_picks_of_a_cache_file(tmp_path, monkeypatch, r, dt, rows, version):
    shape, iters = (30, 40, 72), 3
    gpu = torch.cuda.get_device_name().replace(" ", "_")
    line = f"{version} {gpu} 3 {r} 0 {CODE[dt]} 72 40 30 1 1 16 8 {rows} 16 2" + (" 1" if version == "v2" else "")
    path = tmp_path / "picks"
    path.write_text(line + "\n")
    monkeypatch.setenv("STENCIL_TUNE_CACHE", str(path))
    c, x, want = _problem(3, r, dt, shape, 1, iters)
    s = st.Stencil(3, r, c)
    assert s.default_schedule(shape, CODE[dt]).rows_per_thread == rows
    assert_bits_equal(s.run(x, iters).cpu(), want, line)
    s.close()


@pytest.mark.parametrize("dim,r,shared,sched", [
    (3, 4, False, dict(prefetch=2)), (3, 6, False, dict(t=1, rows_per_thread=2, prefetch=2)),
    (2, 5, False, dict(prefetch=5)), (2, 6, False, dict(t=2, prefetch=6)), (2, 2, True, dict(t=3, prefetch=7)),
    (2, 3, False, dict(t=2, planes_per_step=4, prefetch=10))])
def test_explicit_depths(dim, r, shared, sched):
    shape, iters = ((30, 40, 72) if dim == 3 else (90, 400)), 5
    c, x, want = _problem(dim, r, "f32", shape, 1, iters, shared)
    s = st.Stencil(dim, r, c, shared=shared)
    assert_bits_equal(s.run(x, iters, sched=st.schedule(kernel=st.KERNEL_STREAM, **sched)).cpu(), want, str(sched))
    compiled = st.stencil_resolve_schedule(s.handle, shape[-1], shape[-2], shape[0] if dim == 3 else 1, st.STENCIL_F32,
                                           st.schedule(**{k: v for k, v in sched.items() if k != "prefetch"})).prefetch
    assert_bits_equal(s.run(x, iters, sched=st.schedule(kernel=st.KERNEL_STREAM, **dict(sched, prefetch=compiled))).cpu(),
                      want, f"compiled depth {compiled}")
    with pytest.raises(st.StencilError):
        s.run(x, iters, sched=st.schedule(kernel=st.KERNEL_STREAM, **dict(sched, prefetch=60)))
    s.close()
