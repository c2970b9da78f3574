"""The eigensolver's seed at the edges of its variants: columns of 1 ... 6 x 32 entries in registers, the last size in
shared memory and the first beyond it, odd and even sizes, and matrices the Cholesky factor of a density matrix
does not see: zero, rank one, indefinite and negative blocks.

Bounds: the last refinement correction E has |E_ij| <= 1e-7, what it leaves is of order ||E||^2 <= (n 1e-7)^2, so
that, and n 2^-50 for the rounding of the products, bound the eigenvalues, U diag(lambda) U^dag (both in units
of the block's norm) and U^dag U - 1.
"""
import numpy as np
import pytest

from gpu_util import dev, host, new_ctx

pytestmark = pytest.mark.gpu


def _eig(blocks):
    import torch
    from paper_1103_5391_gb300 import tdmrg as T
    dims = [len(b) for b in blocks]
    ctx = new_ctx()
    try:
        T.tdmrg_set_block(ctx, 0, [(k, 0) for k in range(len(dims))], dims)
        T.tdmrg_set_block(ctx, 1, [(0, 0)], [1])
        ev = torch.full((sum(dims),), np.nan, dtype=torch.float64, device="cuda")
        U = dev(np.full(sum(d * d for d in dims), np.nan))
        T.tdmrg_rho_eig(ctx, dev(np.concatenate([b.ravel() for b in blocks])), ev, U)
        ev, U = ev.cpu().numpy(), host(U)
    finally:
        T.tdmrg_destroy(ctx)
    out, o, e = [], 0, 0
    for d in dims:
        out.append((ev[e:e + d], U[o:o + d * d].reshape(d, d)))
        o, e = o + d * d, e + d
    return out


def _hermitian(rng, lam):
    n = len(lam)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    a = (q * lam) @ q.conj().T
    return (a + a.conj().T) / 2


def _check(blocks):
    for a, (lam, U) in zip(blocks, _eig(blocks)):
        n, big = len(a), max(np.abs(a).max(), 1e-300)
        nrm = big * np.linalg.norm(a / big)      # squares of tiny entries underflow
        tol = (n * 1e-7) ** 2 + n * 2.0 ** -50
        assert np.all(np.diff(lam) <= 0)
        assert np.abs(U.conj().T @ U - np.eye(n)).max() <= tol, n
        assert np.abs(lam - np.linalg.eigvalsh(a)[::-1]).max() <= tol * nrm, n
        assert np.abs((U * lam) @ U.conj().T - a).max() <= tol * nrm, n


@pytest.mark.parametrize("sizes", [(1,), (2, 3), (31, 32, 33), (63, 64, 65), (96, 97), (127, 129), (160, 161), (168, 169), (1, 200, 5)])
def test_sizes(sizes):
    rng = np.random.default_rng(sum(sizes))
    _check([_hermitian(rng, np.exp(-6.0 * (np.arange(n) + rng.random(n)) / n) * 10.0 ** -k) for k, n in enumerate(sizes)])


@pytest.mark.parametrize("kind", ["zero", "rank one", "indefinite", "negative", "tiny"])
@pytest.mark.parametrize("n", [2, 17, 70])
def test_other_matrices(kind, n):
    rng = np.random.default_rng(n)
    x = np.arange(n, dtype=float)
    lam = {"zero": 0 * x, "rank one": np.where(x == 0, 0.7, 0.0), "indefinite": np.cos(2.1 * x + 0.3), "negative": -1.0 - x,
           "tiny": 1e-200 * (1.0 + x)}[kind]
    _check([_hermitian(rng, lam), np.eye(3, dtype=complex)])
