"""roeam_launch_count counts the kernels of roeam_edge_rows and roeam_set_halo, one each."""
import numpy as np
import pytest

import workloads as W
from test_gpu_tile import P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [64, 32])
def test_row_kernels_are_counted(prec):
    spec = W.GridSpec(ni=37, nj=12, dx=0.1, dy=0.1, bc=(W.PERIODIC, W.PERIODIC, 4, W.WALL), params=W.SchemeParams(m_ref=0.5))
    with P().Batch([spec], precision=prec) as b:
        b.set_state(W.random_smooth_state(spec, seed=4), 0)
        n0 = b.launches
        rows = b.edge_rows(0, 2, 0)
        assert b.launches - n0 == 1
        b.set_halo(0, 2, 0, rows)
        assert b.launches - n0 == 2
        assert np.array_equal(rows, b.edge_rows(0, 2, 0))
