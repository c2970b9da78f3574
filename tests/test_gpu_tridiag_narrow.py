"""Lowest Ritz pair of a Lanczos tridiagonal whose other eigenvalues are narrow against one far off (a state pushed up
by a penalty, or the ground state far below): H = s h with the spectrum of h in [-1, 1], one eigenvalue moved to +-1.

Bounds: Lanczos stops at beta <= breakdown_tol (1e-12), and products and orthogonalisation leave 64 nk 2^-53 ||H||, so
the residual of the returned pair is at most r = 1e-12 + 64 nk 2^-53; an eigenvalue is off by no more than the
residual, and the mean of h in the state by r / s.
"""
import numpy as np
import pytest

from gpu_util import dev, host, new_ctx

pytestmark = pytest.mark.gpu
N, NK = 60, 32


@pytest.mark.parametrize("s", [1e-8, 1e-10, 3e-11])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_one_eigenvalue_far_off(s, sign):
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(1)
    q, _ = np.linalg.qr(rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N)))
    h = np.sort(rng.uniform(-1, 1, N))
    lam = s * h
    lam[-1 if sign > 0 else 0] = sign
    H = (q * lam) @ q.conj().T
    H = (H + H.conj().T) / 2
    v = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    ctx = new_ctx(nk_max=NK)
    try:
        T.tdmrg_set_block(ctx, 0, [(0, 0)], [N])
        T.tdmrg_set_block(ctx, 1, [(0, 0)], [1])
        T.tdmrg_set_op(ctx, 0, 0, 0, [((0, 0), (0, 0), H)])
        T.tdmrg_set_hamiltonian(ctx, 0, -1, [])
        x = dev(v)
        e = T.tdmrg_ground_state(ctx, (0, 0), x, nk=NK, restarts=3)
        x = host(x)
    finally:
        T.tdmrg_destroy(ctx)
    r = 1e-12 + 64 * NK * 2.0 ** -53
    w = np.abs(q.conj().T @ x) ** 2
    assert abs(e - lam[0]) <= r
    assert w @ (lam - lam[0]) / w.sum() <= r
