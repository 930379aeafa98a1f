"""FP64 arguments below the normal range, which hardware seeds flush to zero: velocities of 1e-155 (their
squares are subnormal, as in the tail of a Gaussian vortex in still gas) and of 1e-310 (their differences
are). The square root of a subnormal is at most sqrt(2^-1022) = 1.5e-154, so 0 is as good; a slope between
differences whose sum is subnormal is below 1e-308, and 0 as good. Steps against the oracle to the usual
1e-12 of the state's magnitude."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_3d import rel_err3
from test_gpu_tile import P, rel

pytestmark = pytest.mark.gpu


def test_square_root_of_subnormals():
    tiny = np.finfo(np.float64).tiny
    x = np.array([0.0, 5e-324, 1e-320, 1e-310, np.nextafter(tiny, 0), tiny, 4 * tiny])
    assert np.all(np.abs(P().roeam_math_check(x)[:, 2] - np.sqrt(x)) <= np.sqrt(tiny))


def still_gas(speed, shape, seed=3):
    """rho, p varying by 10 %, velocity components of that speed, both signs and equal neighbours among them"""
    r = W.SplitMix64(seed).uniforms(4 * int(np.prod(shape))).reshape((4,) + shape)
    sign = np.floor(3 * r[1:3]) - 1
    return 1 + 0.1 * r[0], speed * sign[0] * (1 + r[1]), speed * sign[1] * (1 + r[2]), 1 + 0.1 * r[3]


@pytest.mark.parametrize("speed", [1e-155, 1e-310])
@pytest.mark.parametrize("recon", [0, 1, 2])
@pytest.mark.parametrize("eps1", [0, 1])
def test_step_of_nearly_still_gas(eps1, recon, speed):
    spec = W.GridSpec(ni=41, nj=23, dx=0.1, dy=0.12, params=W.SchemeParams(m_ref=1e-3, recon=recon, eps1=eps1))
    U = W.prim_to_cons(*still_gas(speed, (spec.nj, spec.ni)))
    dt = 1e-5   # (CFL 0.3 at M_ref = 1e-3; at 1e-3 the oracle's step fails, too)
    with P().Batch([spec], precision=64) as b:
        b.set_state(U, 0)
        b.step(dt_fixed=dt, nsteps=1)
        whole = b.get_state(0)
        b.check()
        b.set_state(U, 0)
        for s in range(3):
            b.stage(s, dt)
        staged = b.get_state(0)
        b.check()
    Uo, _ = oracle.OracleGrid(spec).step(U, dt_fixed=dt)
    assert rel(whole, Uo) <= 1e-12 and rel(staged, Uo) <= 1e-12


@pytest.mark.parametrize("eps1", [0, 1])
def test_3d_step_of_nearly_still_gas(eps1):
    spec = W.GridSpec3(ni=13, nj=9, nk=7, dx=0.1, dy=0.1, dz=0.1, params=W.SchemeParams(m_ref=1e-3, eps1=eps1))
    rho, u, v, p = still_gas(1e-155, (spec.nk, spec.nj, spec.ni))
    U = W.prim_to_cons3(rho, u, v, -u, p)
    with P().Batch3([spec], precision=64) as b:
        b.set_state(U, 0)
        b.step(dt_fixed=1e-5, nsteps=1)
        Ug = b.get_state(0)
        b.check()
    Uo, _ = oracle.OracleGrid3(spec).step(U, dt_fixed=1e-5)
    assert rel_err3(Ug, Uo) <= 1e-12
