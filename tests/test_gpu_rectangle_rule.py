"""Which FP32 grids step in rectangles (one launch a step) and which in strips (three), where one of them
measured at least a fifth faster: single grids, batches of small grids, needles, with and without walls."""
import pytest

import workloads as W
from test_gpu_tile import P, spec_of

pytestmark = pytest.mark.gpu

# (grids, ni, nj, bc, recon, curvilinear, us a step in strips, in rectangles)
MEASURED = [(1, 64, 64, "periodic", 0, False, 11, 5), (1, 256, 256, "periodic", 2, False, 19, 12),
            (1, 400, 400, "box", 1, False, 41, 31), (1, 900, 900, "periodic", 0, False, 46, 68),
            (1, 1000, 1000, "duct", 2, True, 133, 178), (300, 32, 32, "periodic", 0, False, 46, 29),
            (300, 32, 32, "box", 1, False, 109, 56), (300, 32, 32, "duct", 2, True, 145, 66),
            (600, 24, 24, "duct", 2, True, 117, 64), (40, 150, 150, "periodic", 2, False, 84, 112),
            (1, 4, 50000, "periodic", 0, False, 73, 48), (1, 4, 50000, "duct", 2, True, 151, 77),
            (1, 50000, 4, "periodic", 0, False, 28, 45), (1, 50000, 4, "duct", 2, True, 50, 66)]


@pytest.mark.parametrize("count,ni,nj,bc,recon,curv,strips,rectangles", MEASURED)
def test_faster_kernel_is_taken(count, ni, nj, bc, recon, curv, strips, rectangles):
    spec = spec_of(bc, ni, nj, recon, curv=curv)
    with P().Batch([spec] * count, precision=32) as b:
        b.set_states([W.free_stream(spec)] * count)
        n0 = b.launches
        b.step(dt_fixed=1e-5, nsteps=1)
        assert b.launches - n0 == (1 if rectangles < strips else 3)
        b.check()
