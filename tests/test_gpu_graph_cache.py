"""A program that goes round eight (cfl, dt) pairs keeps their graphs, whichever of its two buffers holds the
state when each comes round (from the profiler's record of CUDA calls)."""
import pytest

import workloads as W
from test_gpu_first_calls import recorded
from test_gpu_tile import P, spec_of

pytestmark = pytest.mark.gpu


def test_graphs_of_eight_time_steps_are_kept():
    spec = spec_of("periodic", 40, 33, 0)
    with P().Batch([spec], precision=32) as b:
        U = W.random_smooth_state(spec, seed=2)

        def rounds(n):
            for _ in range(n):
                b.set_state(U, 0)   # (takes a rate slot: the state is in the other buffer when a graph next begins)
                for k in range(8):
                    b.step(dt_fixed=1e-6 * (1 + k), nsteps=12)
        rounds(4)
        names = recorded(lambda: rounds(2))
    assert [n for n in names if "GraphLaunch" in n], sorted(set(names))
    assert not [n for n in names if "GraphInstantiate" in n]
