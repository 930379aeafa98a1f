"""FP64 residuals and norms through the tile kernel, alone and of one grid in a batch: the same bits from the
allocating and the allocation-free call, the oracle's residual to 1e-12 of its magnitude, and norms that are those of that residual (a sum of n squares in another order: relative
rounding far below 1e-13 for these sizes)."""
import numpy as np
import pytest

import oracle
import workloads as W
from test_gpu_tile import P, spec_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recon", [0, 1, 2])
@pytest.mark.parametrize("curv,solid", [(False, False), (True, True)])
def test_residual_and_norms(recon, curv, solid):
    specs = [spec_of("duct" if solid else "periodic", ni, nj, recon, curv=curv, solid=solid) for ni, nj in ((37, 41), (9, 70), (130, 33))]
    Us = [W.random_rough_state(s, seed=5 + k, mach=0.6, jump=0.3) for k, s in enumerate(specs)]
    for batch in ([specs[2]], specs):
        Ub = Us[2:] if len(batch) == 1 else Us
        with P().Batch(batch, precision=64) as b:
            b.set_states(Ub)
            for k, s in enumerate(batch):
                R = b.residual(k)
                S = np.empty_like(R)
                P().roeam_flux_residual_noalloc(b.handle, k, S)
                assert np.array_equal(R, S)
                Ro = oracle.OracleGrid(s).residual(Ub[k])
                assert np.abs(R - Ro).max() <= 1e-12 * np.abs(Ro).max()
                n = s.ni * s.nj - (0 if s.solid is None else int(s.solid.sum()))
                l2, li = b.residual_norm(k, P().ROEAM_NORM_L2), b.residual_norm(k, P().ROEAM_NORM_LINF)
                assert np.allclose(l2, np.sqrt((R ** 2).reshape(4, -1).sum(axis=1) / n), rtol=1e-13, atol=0)
                assert np.array_equal(li, np.abs(R).reshape(4, -1).max(axis=1))
                assert np.array_equal(l2, b.residual_norm(k, P().ROEAM_NORM_L2))
