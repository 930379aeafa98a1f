"""A step gives the same bits whichever kernels run it, walls and solid cells included: rectangles
(roeam_rk_step), strips (roeam_rk_stage) and the host-resident call (strips). And the time-step rate that a
step leaves is that of its result loaded into a new handle."""
import numpy as np
import pytest

import workloads as W
from test_gpu_tile import BCS, P, spec_of

pytestmark = pytest.mark.gpu


def same_bits(spec, U, prec, dt, nsteps=2):
    with P().Batch([spec], precision=prec) as b, P().Batch([spec], precision=prec) as q, P().Batch([spec], precision=prec) as h:
        b.set_state(U, 0)
        q.set_state(U, 0)
        n0 = b.launches
        b.step(dt_fixed=dt, nsteps=nsteps)
        assert b.launches - n0 == nsteps * (1 if prec == 32 else 3)
        for _ in range(nsteps):
            for s in range(3):
                q.stage(s, dt)
        Ub = b.get_state(0)
        assert np.array_equal(Ub, q.get_state(0))
        out = np.empty_like(U)
        P().roeam_step_host(h.handle, 0.0, dt, nsteps, np.ascontiguousarray(U), out)
        assert np.array_equal(Ub, out)
        assert np.array_equal(b.max_rate(), q.max_rate()) and np.array_equal(b.max_rate(), h.max_rate())
        with P().Batch([spec], precision=prec) as n:
            n.set_state(Ub, 0)
            assert np.array_equal(b.max_rate(), n.max_rate())


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("recon", [0, 1, 2])
@pytest.mark.parametrize("bc", sorted(BCS))
def test_rectangles_and_strips_give_the_same_bits(bc, recon, prec):
    for ni, nj in ((4, 4), (12, 9), (37, 41), (90, 66), (130, 7)):
        for curv in (False, True):
            for solid in (False, True):
                if solid and (W.PERIODIC in BCS[bc] or min(ni, nj) < 9):
                    continue
                spec = spec_of(bc, ni, nj, recon, curv=curv, solid=solid, eps1=(ni + nj) % 2)
                same_bits(spec, W.random_rough_state(spec, seed=ni + 100 * nj, mach=0.7, jump=0.3), prec, 0.01)


@pytest.mark.parametrize("recon", [1, 2])
@pytest.mark.parametrize("curv", [False, True])
def test_same_bits_across_marginal_jumps(curv, recon):
    """Six orders of magnitude in rho and p next to walls and solid cells, where FP32 decides faces in FP64."""
    spec = spec_of("box", 45, 38, recon, curv=curv, solid=True)
    U = W.random_rough_state(spec, seed=5, mach=0.3, jump=0.2)
    U[:, 10:20, 12:30] *= 1e-6
    U[:, :2, :] *= 1e-6
    for prec in (32, 64):
        same_bits(spec, U, prec, 1e-8)
