"""FP64 loads from device memory: queued back to back they take no longer than waited for one by one, and a
state of 128^2 cells is loaded about as fast as one of 32^2 (their rates are spread over the processors)."""
import time

import numpy as np
import pytest

import workloads as W
from test_gpu_tile import P, spec_of

pytestmark = pytest.mark.gpu


def times(spec, wait, prec=64):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    U = torch.tensor(W.random_smooth_state(spec, seed=1, mach=0.3), device="cuda")
    with P().Batch([spec], precision=prec) as b:
        best = 1e9
        for _ in range(10):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(30):
                b.set_state_device(U, 0, stream)
                if wait:
                    torch.cuda.synchronize()
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        assert np.array_equal(b.get_state(0), U.cpu().numpy())
    return best


@pytest.mark.parametrize("n", [64, 128, 256])
def test_queued_loads_are_not_slower(n):
    spec = spec_of("periodic", n, n, 0)
    for _ in range(6):   # (another process on the GPU may disturb one side)
        queued, alone = times(spec, False), times(spec, True)
        if queued <= alone:
            return
    assert queued <= alone


def test_small_loads_are_spread():
    for _ in range(6):
        large, small = times(spec_of("periodic", 128, 128, 0), False), times(spec_of("periodic", 16, 16, 0), False)
        if large <= 1.6 * small:
            return
    assert large <= 1.6 * small
