"""CUDA work beyond the kernels, from the profiler's record: the first load and step of a handle that runs in
rectangles clear no rate slots (roeam_create_grid left them zero)."""
import pytest

import workloads as W
from test_gpu_tile import P, spec_of

pytestmark = pytest.mark.gpu


def recorded(fn):
    import torch
    from torch.profiler import ProfilerActivity, profile
    kinds = [ProfilerActivity.CPU, ProfilerActivity.CUDA]
    with profile(activities=kinds):   # (the first session of a process records nothing)
        torch.zeros(8, device="cuda").add_(1)
        torch.cuda.synchronize()
    with profile(activities=kinds) as prof:
        fn()
        torch.cuda.synchronize()
    names = [e.name for e in prof.events()]
    if not any("kernel" in n for n in names):
        pytest.skip("the profiler records no GPU work here")
    return names


@pytest.mark.parametrize("prec", [64, 32])
def test_first_load_and_step_clear_nothing(prec):
    spec = spec_of("periodic", 40, 33, 0)
    U = W.random_smooth_state(spec, seed=2)
    with P().Batch([spec], precision=prec) as b:
        def first():
            b.set_state(U, 0)
            b.step(cfl=0.4, nsteps=1)
            b.get_state(0)
        names = recorded(first)
    assert any("tile_kernel" in n for n in names), names
    assert not [n for n in names if "memset" in n.lower()]
