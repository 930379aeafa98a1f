"""Where every warp has a unit or less, shapes that claim units dynamically run as those that do not: equal
times (claims once cost a 64^2 step's three stages 16.5 us against 12.3) and equal bits."""
import time

import numpy as np
import pytest

import workloads as W
from test_gpu_tile import P, spec_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recon,curv", [(0, False), (2, False), (2, True)])
def test_no_claims_where_units_are_few(recon, curv):
    import torch
    spec = spec_of("periodic", 64, 64, recon, curv=curv)
    U = W.random_smooth_state(spec, seed=1, mach=0.3)
    with P().Batch([spec], precision=32) as b:
        def run(cfg):
            b.set_tile_config(cfg)
            b.set_state(U, 0)
            best = 1e9
            for _ in range(8):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                for _ in range(20):
                    for s in range(3):
                        b.stage(s, 1e-4)
                torch.cuda.synchronize()
                best = min(best, time.perf_counter() - t0)
            return best, b.get_state(0)
        for _ in range(6):   # (another process on the GPU may disturb one side)
            (claiming, U0), (static, U1) = run(0), run(5)
            assert np.array_equal(U0, U1)
            if claiming <= 1.1 * static:
                return
    assert claiming <= 1.1 * static
