"""Reading a large state into device memory is faster than loading it (which also takes the time-step rates);
with 1024 blocks it was not. Grids of all sizes come back as loaded."""
import time

import numpy as np
import pytest

import workloads as W
from test_gpu_tile import P

pytestmark = pytest.mark.gpu


def test_large_read():
    import torch
    s = W.GridSpec(ni=3000, nj=3000, dx=0.1, dy=0.1, params=W.SchemeParams(m_ref=0.5))
    stream = torch.cuda.current_stream().cuda_stream
    U = torch.tensor(W.free_stream(s), device="cuda")
    V = torch.empty_like(U)
    with P().Batch([s], precision=32) as b:
        b.set_state_device(U, 0, stream)

        def best(fn):
            t = []
            for _ in range(20):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                for _ in range(5):
                    fn()
                torch.cuda.synchronize()
                t.append(time.perf_counter() - t0)
            return min(t)
        for _ in range(6):   # (another process on the GPU may disturb one side)
            read, load = best(lambda: b.get_state_device(V, 0, stream)), best(lambda: b.set_state_device(U, 0, stream))
            if read <= 0.95 * load:
                break
        assert read <= 0.95 * load
        assert torch.equal(V, U.float().double())


@pytest.mark.parametrize("prec", [64, 32])
def test_reads_of_uneven_batches(prec):
    specs = [W.GridSpec(ni=a, nj=b, dx=0.1, dy=0.1, params=W.SchemeParams(m_ref=0.5))
             for a, b in [(4, 4), (1100, 1000), (33, 5)] + [(9, 8)] * 9]
    Us = [W.random_smooth_state(s, seed=2 + k, mach=0.2).astype(np.float32).astype(np.float64) for k, s in enumerate(specs)]
    with P().Batch(specs, precision=prec) as b:
        b.set_states(Us)
        assert all(np.array_equal(x, y) for x, y in zip(b.get_states(), Us))
        assert np.array_equal(b.get_state(1), Us[1])
