"""roeam_autotune on handles whose steps run in rectangles (FP64; small FP32 grids): the shapes apply to the
strip kernels, so the trials run those, three launches a step (a step in rectangles is one launch in
FP32), and steps, state and launches are afterwards what they were."""
import numpy as np
import pytest

import workloads as W
from test_gpu_tile import P, spec_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [64, 32])
def test_trials_run_what_the_shapes_apply_to(prec):
    spec = spec_of("periodic", 71, 53, 0, use_s1=prec == 32)   # (a workload per precision of its own)
    U = W.random_smooth_state(spec, seed=11, mach=0.4, amp=0.3)
    steps = 9   # (a graph among them)
    with P().Batch([spec], precision=prec) as b, P().Batch([spec], precision=prec) as q:
        b.set_state(U, 0)
        q.set_state(U, 0)
        n0 = b.launches
        best, ms = b.autotune(0.4, steps)
        assert ms[best] == ms.min()
        # (every shape ends up at two rows here: two layouts, claiming and static, each timed twice)
        assert b.launches - n0 == 2 * 2 * (1 + steps) * 3
        for n in (1, 9, 2):
            n0 = b.launches
            db, dq = (x.step(cfl=0.4, nsteps=n, want_dt=True) for x in (b, q))
            assert b.launches - n0 == n * (1 if prec == 32 else 3)
            assert np.array_equal(db, dq) and np.array_equal(b.get_state(0), q.get_state(0))
