"""Blocks of a density matrix that are zero (a sector no target reaches) or real (the real-basis variant): a zero block
has the unit vectors as eigenvectors and zero eigenvalues, exactly, whatever its neighbours; a real symmetric block
has eigenvectors without imaginary part, exactly.

Sizes on either side of the limits of the seed's variants: one CTA with 1 to 4 steps of 16 rows in registers up to 64
columns, a cluster of four CTAs with 2 or 3 steps up to 160, the factor in global memory beyond.  Bounds of the real
blocks: the last refinement correction leaves at most (n 1e-7)^2, the products n 2^-50.
"""
import numpy as np
import pytest

from test_gpu_eig_seed import _eig

pytestmark = pytest.mark.gpu


def _real_block(rng, n):
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    a = (q * np.exp(-6.0 * (np.arange(n) + rng.random(n)) / n)) @ q.T
    return ((a + a.T) / 2).astype(complex)


@pytest.mark.parametrize("n", [1, 2, 16, 17, 48, 64, 65, 128, 129, 160, 161])
def test_zero_block(n):
    rng = np.random.default_rng(n)
    zero = np.zeros((n, n), complex)
    for lam, U in _eig([zero, _real_block(rng, 20), zero])[::2]:
        assert not lam.any()
        assert np.array_equal(U, np.eye(n))


@pytest.mark.parametrize("n", [2, 16, 17, 48, 64, 65, 128, 129, 160, 161])
def test_real_block(n):
    rng = np.random.default_rng(100 + n)
    blocks = [_real_block(rng, n), np.zeros((n, n), complex), _real_block(rng, 33)]
    out = _eig(blocks)
    for lam, U in out:
        assert not U.imag.any()
    lam, U = out[0]
    tol = (n * 1e-7) ** 2 + n * 2.0 ** -50
    assert np.abs(U.conj().T @ U - np.eye(n)).max() <= tol
    assert np.abs((U * lam) @ U.conj().T - blocks[0]).max() <= tol * np.linalg.norm(blocks[0])
