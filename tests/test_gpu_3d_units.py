"""The 3D stage kernels at the edges of their work units: FP32 marches tiles of 30 x 14 columns over
segments of planes, FP64 rectangles and segments that an estimate chooses, so extents around multiples of
those, thin grids, every boundary kind on each side and 0 to 3 scalars (tails of 1, 2, 4 and 4 values)
against the oracle; the residual, a reload and a second handle in between."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

TOL = {64: 1e-12, 32: 1e-5}


def P():
    import paper_1711_09272_gb300 as pkg
    return pkg


def rel(Ug, Uo):
    m = np.sqrt(Uo[1] ** 2 + Uo[2] ** 2 + Uo[3] ** 2).max()
    sc = np.array([np.abs(Uo[0]).max(), m, m, m, np.abs(Uo[4]).max()] + [np.abs(Uo[v]).max() for v in range(5, len(Uo))])
    return float(np.max(np.abs(Ug - Uo).reshape(len(Uo), -1).max(axis=1) / sc))


BCS = {"periodic": (W.PERIODIC,) * 6,
       "channel": (W.INFLOW, W.OUTFLOW, W.WALL, W.WALL, W.PERIODIC, W.PERIODIC),
       "box": (W.WALL,) * 6,
       "mixed": (W.OUTFLOW, W.WALL, W.PERIODIC, W.PERIODIC, W.INFLOW, W.WALL)}
SIZES = [(1, 1, 9), (2, 33, 5), (30, 14, 7), (31, 15, 1), (61, 29, 4), (9, 7, 40), (95, 3, 6)]


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("bc", sorted(BCS))
def test_unit_edges(bc, prec):
    for n, (ni, nj, nk) in enumerate(SIZES):
        ns = n % 4
        spec = W.GridSpec3(ni=ni, nj=nj, nk=nk, dx=0.05, dy=0.06, dz=0.07, bc=BCS[bc], nscal=ns,
                           inflow=(1.2, 0.7, 0.1, -0.2, 1.1) + (0.4, 0.1, 0.9)[:ns],
                           params=W.SchemeParams(m_ref=0.5, eps1=n % 2, use_s1=0 if n == 3 else 1))
        U = W.random_rough_state3(spec, seed=31 + n, mach=0.8, jump=0.3)
        with P().Batch3([spec], precision=prec) as b:
            b.set_state(U, 0)
            U0 = b.get_state(0)
            R = b.residual(0)
            b.step(0.4, nsteps=2)
            U2 = b.get_state(0)
            b.set_state(U0, 0)
            b.step(0.4, nsteps=2)
            assert np.array_equal(b.get_state(0), U2)
        o = oracle.OracleGrid3(spec)
        Uo, _ = o.step(U0, cfl=0.4, nsteps=2)
        assert rel(U2, Uo) <= 2 * TOL[prec], (ni, nj, nk)
        Ro = o.residual(U0)
        assert np.abs(R - Ro).max() <= (1e-12 if prec == 64 else 2e-5) * np.abs(Ro).max() + (1e-12 if prec == 64 else 1e-4)
