"""Orthonormal eigenvectors of density matrices whose spectra span more than the range of FP64 (20 and 30 decades, as in
long DMRG blocks), several sectors side by side, complex and real: a close pair far below the largest eigenvalue is
coupled by rounding only, and turning it must not cost the orthonormality that truncation and renormalisation rely on.
Exact multiplets over twelve decades: their states may be mixed at will, and must not be coupled to others by it.

Bounds: an iteration leaves at most (n 1e-7)^2, the products n 2^-50; eigenvalues in units of ||rho||.
A last correction of |E| <= 8e-7 formed in FP32 leaves 8e-7 2^-23 a product term: n 2^-43 for the reconstruction.
"""
import numpy as np
import pytest

from test_gpu_eig_seed import _eig

pytestmark = pytest.mark.gpu
SIZES = (12, 20, 33, 47, 60)


@pytest.mark.parametrize("decades", [14, 20, 30])
@pytest.mark.parametrize("seed", range(8))
def test_orthonormal(decades, seed):
    rng = np.random.default_rng(1000 * seed + 12)
    blocks = []
    for n in SIZES:
        z = rng.standard_normal((n, n)) + (0 if seed % 2 else 1j * rng.standard_normal((n, n)))
        q, _ = np.linalg.qr(z)
        a = (q * 10.0 ** (-decades * (np.arange(n) + rng.random(n)) / n)) @ q.conj().T
        blocks.append((a + a.conj().T).astype(complex) / 2)
    for a, (lam, U) in zip(blocks, _eig(blocks)):
        n, tol = len(a), (len(a) * 1e-7) ** 2 + len(a) * 2.0 ** -50
        assert np.abs(U.conj().T @ U - np.eye(n)).max() <= tol, n
        assert np.abs(lam - np.linalg.eigvalsh(a)[::-1]).max() <= tol * np.linalg.norm(a), n


@pytest.mark.parametrize("sizes", [SIZES, (170, 200)])
@pytest.mark.parametrize("seed", range(8))
def test_multiplets(sizes, seed):
    rng = np.random.default_rng(1000 * seed + sizes[0])
    blocks = []
    for n in sizes:
        z = rng.standard_normal((n, n)) + (0 if seed % 2 else 1j * rng.standard_normal((n, n)))
        q, _ = np.linalg.qr(z)
        a = (q * np.resize(10.0 ** (-12 * rng.random(n // 4)), n)) @ q.conj().T
        blocks.append((a + a.conj().T).astype(complex) / 2)
    for a, (lam, U) in zip(blocks, _eig(blocks)):
        n, nrm = len(a), np.linalg.norm(a)
        assert np.abs(U.conj().T @ U - np.eye(n)).max() <= (n * 1e-7) ** 2 + n * 2.0 ** -50, n
        assert np.linalg.norm((U * lam) @ U.conj().T - a) <= n * 2.0 ** -43 * nrm, n
