"""Lanczos on H = offset + s h, the spectrum of h in [-1, 1], s as small as 3e-11: every product is the old vector to seven
or more digits, and the orthogonalisation has to find the rest.  The Krylov space is that of h, so the lowest Ritz pair
of one run is that of a plain Lanczos on h in numpy: offset + s theta.  Vectors of one block, of several blocks staged
in shared memory (60 x 40), and of more elements per block than that holds (600 x 400).  Segmented advance: such a problem
beside an ordinary one takes all its steps.

Bounds: products and orthogonalisation leave a residual of r = 64 nk 2^-53 |offset| in the Lanczos relation; the Ritz value
is off by as much, and the vector by r over the gap s (theta_1 - theta_0).
"""
import numpy as np
import pytest

from gpu_util import dev, host, new_ctx
from test_gpu_tridiag_min import _lanczos

pytestmark = pytest.mark.gpu
NK = 20


def _hermitian(rng, n):
    q, _ = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    a = (q * rng.uniform(-0.5, 0.5, n)) @ q.conj().T
    return (a + a.conj().T) / 2


def _load(T, ctx, A, B, offset, s):
    T.tdmrg_set_block(ctx, 0, [(0, 0)], [len(A)])
    T.tdmrg_set_block(ctx, 1, [(0, 0)], [len(B)])
    T.tdmrg_set_op(ctx, 0, 0, 0, [((0, 0), (0, 0), offset * np.eye(len(A)) + s * A)])
    T.tdmrg_set_op(ctx, 1, 0, 0, [((0, 0), (0, 0), s * B)])
    T.tdmrg_set_hamiltonian(ctx, 0, 0, [])


class _Sum:
    """h = A (x) 1 + 1 (x) B on row-major vectors"""

    def __init__(self, A, B):
        self.A, self.B = A, B

    def __matmul__(self, v):
        x = v.reshape(len(self.A), len(self.B))
        return (self.A @ x + x @ self.B.T).ravel()


@pytest.mark.parametrize("dims", [(60, 1), (60, 40), (600, 400)])
@pytest.mark.parametrize("offset", [1.0, -1.0])
@pytest.mark.parametrize("s", [1.0, 1e-6, 1e-8, 1e-10, 3e-11])
def test_ritz_pair(dims, offset, s):
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(dims[1])
    A, B = _hermitian(rng, dims[0]), _hermitian(rng, dims[1])
    v = rng.standard_normal(dims[0] * dims[1]) + 1j * rng.standard_normal(dims[0] * dims[1])
    ctx = new_ctx(nk_max=32)
    try:
        _load(T, ctx, A, B, offset, s)
        x = dev(v)
        e = T.tdmrg_ground_state(ctx, (0, 0), x, nk=NK, restarts=1)
        x = host(x)
    finally:
        T.tdmrg_destroy(ctx)
    theta, want = _lanczos(_Sum(A, B), v, NK)
    r = 64 * NK * 2.0 ** -53 * (1 + s)
    assert abs(e - (offset + s * theta[0])) <= r
    assert np.linalg.norm(x - want * np.vdot(want, x)) <= r / (s * (theta[1] - theta[0]))
    assert abs(np.linalg.norm(x) - 1) <= r / s


def test_segments():
    import torch
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(3)
    jobs, big = [], new_ctx(nk_max=32)
    try:
        for n, offset, s in [(60, 1.0, 1e-8), (50, 0.0, 1.0), (70, 2.0, 1e-9)]:
            ctx = new_ctx(nk_max=32)
            _load(T, ctx, _hermitian(rng, n), np.zeros((1, 1)), offset, s)
            jobs.append((n, ctx))
        Q, off = T.tdmrg_direct_sum(big, [c for _, c in jobs], [(0, 0)] * 3)
        phi = dev(rng.standard_normal(off[-1]) + 1j * rng.standard_normal(off[-1]))
        out = [torch.zeros_like(phi) for _ in range(2)]
        T.tdmrg_evolve_segments(big, Q, phi, [n for n, _ in jobs], [0.0, 1e-3], NK, out)
        nk, _ = T.tdmrg_evolve_segments_info(big, Q, NK, 3)
        assert list(nk) == [NK] * 3
    finally:
        T.tdmrg_destroy(big)
        for _, c in jobs:
            T.tdmrg_destroy(c)
