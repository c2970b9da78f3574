"""Lowest Ritz pair of one Lanczos run (tdmrg_ground_state with one restart) against a plain Lanczos in numpy, for
Krylov dimensions from 2 to 32, a start vector that is already an eigenvector (breakdown at one vector), spectra
of either sign, far from and around zero, and a tiny and a large scale.

Bounds: both sides build their tridiagonal with errors of order nk 2^-53 ||H||, which moves the Ritz value by as
much and turns the Ritz vector by that over the gap to the next Ritz value; the factor 64 covers the sums.
"""
import numpy as np
import pytest

from gpu_util import dev, host, new_ctx

pytestmark = pytest.mark.gpu
N = 60


def _lanczos(H, v, nk):
    V, a, b = [v / np.linalg.norm(v)], [], []
    for j in range(nk):
        w = H @ V[-1]
        a.append(np.vdot(V[-1], w).real)
        for _ in range(2):
            for u in V:
                w = w - np.vdot(u, w) * u
        if j + 1 < nk:
            b.append(np.linalg.norm(w))
            V.append(w / b[-1])
    lam, S = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
    return lam, np.array(V).T @ S[:, 0]


def _run(H, v, nk):
    from paper_1103_5391_gb300 import tdmrg as T
    ctx = new_ctx(nk_max=32)
    try:
        T.tdmrg_set_block(ctx, 0, [(0, 0)], [len(H)])
        T.tdmrg_set_block(ctx, 1, [(0, 0)], [1])
        T.tdmrg_set_op(ctx, 0, 0, 0, [((0, 0), (0, 0), H)])
        T.tdmrg_set_hamiltonian(ctx, 0, -1, [])
        x = dev(v)
        e = T.tdmrg_ground_state(ctx, (0, 0), x, nk=nk, restarts=1)
        return e, host(x)
    finally:
        T.tdmrg_destroy(ctx)


def _matrix(rng, shift, scale):
    q, _ = np.linalg.qr(rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N)))
    H = (q * (shift + np.sort(rng.uniform(-1, 1, N)))) @ q.conj().T
    return scale * (H + H.conj().T) / 2


@pytest.mark.parametrize("nk", [2, 3, 5, 16, 31, 32])
@pytest.mark.parametrize("shift,scale", [(0.0, 1.0), (3.0, 1.0), (-2.0, 1e3), (1.0, 1e-9)])
def test_ritz_pair(nk, shift, scale):
    rng = np.random.default_rng(nk)
    H = _matrix(rng, shift, scale)
    v = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    lam, want = _lanczos(H, v, nk)
    e, got = _run(H, v, nk)
    nrm = np.linalg.norm(H, 2)
    tol = 64 * nk * 2.0 ** -53 * nrm
    assert abs(e - lam[0]) <= tol
    assert abs(np.linalg.norm(got) - 1) <= 64 * nk * 2.0 ** -53
    assert np.linalg.norm(got - want * np.vdot(want, got)) <= tol / (lam[1] - lam[0])


def test_start_is_an_eigenvector():
    rng = np.random.default_rng(7)
    H = np.diag(rng.uniform(-1, 1, N)).astype(complex)
    v = np.zeros(N, complex)
    v[11] = 2.0
    e, got = _run(H, v, 16)
    assert abs(e - H[11, 11].real) <= 64 * 2.0 ** -53
    assert np.abs(np.abs(got) - (np.arange(N) == 11)).max() <= 64 * 2.0 ** -53
