"""The tile kernels (a whole SSP-RK3 step per launch in FP32 on grids too small to fill the chip with
warp strips, a stage per launch in FP64): against the oracle and against the strip kernels
(roeam_rk_stage runs them on the same grid) over sizes around the rectangles' edges, every boundary
kind, walls and solid cells next to rectangle edges, curvilinear geometry and both reconstructions;
several steps (the state then alternates between two buffers, and eight steps go through a graph)
with reads and writes of the state in between."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

TOL = {64: 1e-12, 32: 1e-5}   # per step, of the state's magnitude


def P():
    import paper_1711_09272_gb300 as pkg
    return pkg


def rel(Ug, Uo):
    m = np.sqrt(Uo[1] ** 2 + Uo[2] ** 2).max()
    sc = np.array([np.abs(Uo[0]).max(), m, m, np.abs(Uo[3]).max()])
    return float(np.max(np.abs(Ug - Uo).reshape(4, -1).max(axis=1) / sc))


BCS = {"periodic": (W.PERIODIC,) * 4, "duct": (W.INFLOW, W.OUTFLOW, W.WALL, W.WALL),
       "box": (W.WALL,) * 4, "mixed": (W.WALL, W.INFLOW, W.OUTFLOW, W.INFLOW),
       "x_periodic": (W.PERIODIC, W.PERIODIC, W.WALL, W.OUTFLOW), "y_periodic": (W.OUTFLOW, W.WALL, W.PERIODIC, W.PERIODIC)}


def spec_of(bc, ni, nj, recon, curv=False, solid=False, **p):
    s = W.GridSpec(ni=ni, nj=nj, dx=0.1, dy=0.12, bc=BCS[bc], inflow=(1.1, 0.5, 0.1, 0.9),
                   params=W.SchemeParams(m_ref=0.5, recon=recon, **p))
    if curv:
        X, Y = np.meshgrid(np.arange(ni + 1) * s.dx, np.arange(nj + 1) * s.dy)
        w = np.sin(2 * np.pi * np.arange(ni + 1) / ni)[None, :] * np.sin(2 * np.pi * np.arange(nj + 1) / nj)[:, None]
        s.xv, s.yv = X + 0.15 * s.dx * w, Y + 0.15 * s.dy * w
    if solid:
        s.solid = np.zeros((nj, ni), np.uint8)
        s.solid[nj // 3:nj // 2 + 1, ni // 3:ni // 2 + 1] = 1
        s.solid[: max(1, nj // 5), ni - max(1, ni // 4):] = 1
    return s


def check_against_strips_and_oracle(spec, U, prec, cfl=0.4):
    with P().Batch([spec], precision=prec) as b, P().Batch([spec], precision=prec) as q:
        b.set_state(U, 0)
        q.set_state(U, 0)
        U0 = b.get_state(0)
        l0 = b.launches
        dt = b.step(cfl=cfl, nsteps=1, want_dt=True)[0]
        assert b.launches - l0 == (1 if prec == 32 else 3)
        Ut = b.get_state(0)
        for s in range(3):
            q.stage(s, dt)
        Us = q.get_state(0)
        assert np.array_equal(b.max_rate(), b.max_rate()) and b.max_rate()[0] == pytest.approx(q.max_rate()[0], rel=TOL[prec])
    Uo, _ = oracle.OracleGrid(spec).step(U0, cfl=cfl)
    assert rel(Ut, Uo) <= TOL[prec]
    assert rel(Ut, Us) <= TOL[prec]


SIZES = [(4, 4), (5, 9), (31, 4), (33, 34), (64, 65), (130, 7), (7, 131), (97, 89)]


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("recon", [0, 1, 2])
@pytest.mark.parametrize("bc", sorted(BCS))
def test_one_step_cartesian(bc, recon, prec):
    for ni, nj in SIZES:
        spec = spec_of(bc, ni, nj, recon, eps1=(ni + nj) % 2, use_s1=0 if ni == 33 else 1)
        check_against_strips_and_oracle(spec, W.random_rough_state(spec, seed=ni + 100 * nj, mach=0.8, jump=0.3), prec)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("recon", [0, 2])
@pytest.mark.parametrize("bc", sorted(BCS))
def test_one_step_curvilinear_and_solid(bc, recon, prec):
    for ni, nj in ((12, 9), (37, 41), (90, 66)):
        periodic = W.PERIODIC in BCS[bc]
        for curv, solid in ((True, False), (False, True), (True, True)):
            if solid and periodic:
                continue
            spec = spec_of(bc, ni, nj, recon, curv=curv, solid=solid)
            check_against_strips_and_oracle(spec, W.random_rough_state(spec, seed=7 + ni, mach=0.7, jump=0.3), prec)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("recon", [0, 1])
def test_several_steps_batch_and_restart(recon, prec):
    """A batch of uneven grids over 1 + 9 + 3 steps (odd counts leave the state in the other buffer,
    nine include a graph), a restart from the state read back half way: bit for bit the same."""
    specs = [spec_of("periodic", 40, 23, recon), spec_of("periodic", 9, 70, recon), spec_of("duct", 31, 33, recon)]
    Us = [W.random_smooth_state(s, seed=3 + k, mach=0.4, amp=0.3) for k, s in enumerate(specs)]
    with P().Batch(specs, precision=prec) as b, P().Batch(specs, precision=prec) as q:
        b.set_states(Us)
        U0 = b.get_states()
        for n in (1, 9):
            b.step(cfl=0.4, nsteps=n)
        half = b.get_states()
        q.set_states(half)
        db, dq = (x.step(cfl=0.4, nsteps=3, want_dt=True) for x in (b, q))
        assert np.array_equal(db, dq)
        end, again = b.get_states(), q.get_states()
        R = [b.residual(k) for k in range(3)]
        b.check()
    for k, s in enumerate(specs):
        assert np.array_equal(end[k], again[k])
        Uo, _ = oracle.OracleGrid(s).step(U0[k], cfl=0.4, nsteps=13)
        assert rel(end[k], Uo) <= 13 * TOL[prec]
        assert np.isfinite(R[k]).all()


def test_marginal_jumps_fp32():
    """Faces across six orders of magnitude in rho and p (decided in FP64 on their own), at a time
    step that keeps the thin region's state positive."""
    spec = spec_of("box", 45, 38, 2)
    U = W.random_rough_state(spec, seed=5, mach=0.3, jump=0.2)
    U[:, 10:20, 12:30] *= 1e-6
    check_against_strips_and_oracle(spec, U, 32, cfl=1e-7)


def test_device_errors_are_reported():
    spec = spec_of("periodic", 30, 30, 0)
    U = W.random_smooth_state(spec, seed=2)
    for bad, status in ((-1.0, 4), (np.nan, 5)):
        V = U.copy()
        V[3, 11, 12] = bad
        with P().Batch([spec], precision=32) as b:
            b.set_state(V, 0)
            b.step(cfl=0.4, dt_fixed=1e-4, nsteps=1)
            with pytest.raises(P().RoeamError) as e:
                b.check()
            assert e.value.status == status
            b.set_state(U, 0)
            b.step(cfl=0.4, nsteps=2)
            b.check()
