"""The targets of a Krylov advance as linear combinations of the basis: one to sixteen of them, vectors around the 128
elements of a block, Krylov dimensions that are no multiple of four.

Every target of a joint call equals the same target asked for alone: the coefficients come from the same tridiagonal
(its exponential, a Taylor series on substeps, is within 1e-14 of the exact one for either list of times) and each
component is a sum of at most nk terms with 4 roundings, so the difference is below (2e-14 + 8 nk 2^-53) |phi| < 1e-13 |phi|.
"""
import numpy as np
import pytest

from gpu_util import dev, host, new_ctx
from workloads import sectors as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,m,nk,n_v", [(8, 4, 5, 1), (8, 8, 6, 3), (8, 24, 7, 16), (12, 60, 10, 9), (16, 120, 11, 4)])
def test_targets_alone_and_together(L, m, nk, n_v):
    from paper_1103_5391_gb300 import problem, tdmrg as T
    ss = S.make_synthetic(L, m, 4.0, nbonds=1, seed=5)
    ctx = new_ctx()
    try:
        problem.load_synthetic(ctx, ss)
        n = T.tdmrg_sector_size(ctx, ss.Q0)
        rng = np.random.default_rng(L + m)
        x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
        phi = dev(x)
        times = [0.01 + 0.003 * k * k for k in range(n_v)]
        outs = [dev(np.full(n, np.nan + 0j)) for _ in range(n_v)]
        T.tdmrg_evolve(ctx, ss.Q0, phi, times, nk, outs)
        got = [host(o) for o in outs]
        for k in range(n_v):
            alone = dev(np.full(n, np.nan + 0j))
            T.tdmrg_evolve(ctx, ss.Q0, phi, [times[k]], nk, [alone])
            assert np.abs(got[k] - host(alone)).max() < 1e-13 * np.linalg.norm(x)
    finally:
        T.tdmrg_destroy(ctx)
