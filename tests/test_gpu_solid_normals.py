"""Reconstruction next to solid cells on a curvilinear grid: a solid stencil cell is replaced by the
mirror of the adjacent fluid cell about their common face, whose normal differs from the next row's.
One stage (residual) and one step of the strip kernels (stage calls) against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("recon", [1, 2])
def test_mirror_normals_above_and_below_solids(recon, prec):
    import paper_1711_09272_gb300 as P
    ni, nj = 12, 9
    X, Y = np.meshgrid(np.arange(ni + 1) * 0.1, np.arange(nj + 1) * 0.12)
    w = np.sin(2 * np.pi * np.arange(ni + 1) / ni)[None, :] * np.sin(2 * np.pi * np.arange(nj + 1) / nj)[:, None]
    solid = np.zeros((nj, ni), np.uint8)
    solid[3:5, 4:7] = 1
    solid[:1, 9:] = 1
    spec = W.GridSpec(ni=ni, nj=nj, dx=0.1, dy=0.12, bc=(W.WALL,) * 4, xv=X + 0.015 * w, yv=Y + 0.018 * w, solid=solid,
                      params=W.SchemeParams(m_ref=0.5, recon=recon))
    U = W.random_rough_state(spec, seed=19, mach=0.7, jump=0.3)
    with P.Batch([spec], precision=prec) as b:
        b.set_state(U, 0)
        U0 = b.get_state(0)
        dt = 0.4 / b.max_rate()[0]
        for s in range(3):
            b.stage(s, dt)
        U1 = b.get_state(0)
    Uo, _ = oracle.OracleGrid(spec).step(U0, cfl=0.4, dt_fixed=dt)
    m = np.sqrt(Uo[1] ** 2 + Uo[2] ** 2).max()
    sc = np.array([np.abs(Uo[0]).max(), m, m, np.abs(Uo[3]).max()])
    assert np.max(np.abs(U1 - Uo).reshape(4, -1).max(axis=1) / sc) <= {64: 1e-12, 32: 1e-5}[prec]
