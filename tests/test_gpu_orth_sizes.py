"""The Lanczos orthogonalisation around the sizes where its block split and its shared-memory staging change: vectors of
one element up to several blocks, one block per SM exactly full, slices of which only some Krylov vectors fit in shared
memory and slices of which none do, breakdown in the middle of a run, segments of very different lengths next to each
other (some empty of work, one stopping at once).  A diagonal H makes H v exact, so that V, alpha and beta depend on the
orthogonalisation alone.

Bounds: the targets of an advance are V c with |c| = |phi|; V is orthonormal and spans the Krylov space to rounding, so
the exact exponential of the diagonal H on a vector with few distinct eigenvalues (an invariant subspace of at most nk
dimensions) is reached to nk^2 2^-50 |phi|.
"""
import numpy as np
import pytest

from gpu_util import dev, host, new_ctx

pytestmark = pytest.mark.gpu


def _ctx(T, lam, **kw):
    """H = diag(lam) as one left sector per run of equal eigenvalues x a right sector (dimension d_k x 1)."""
    ctx = new_ctx(nk_max=32, **kw)
    dims, vals = [], []
    for v, d in lam:
        dims.append(d)
        vals.append(v)
    n = len(dims)
    T.tdmrg_set_block(ctx, 0, [(k, 0) for k in range(n)], [1] * n)
    T.tdmrg_set_block(ctx, 1, [(k, 0) for k in range(n)], dims[::-1])
    T.tdmrg_set_op(ctx, 0, 0, 0, [((k, 0), (k, 0), np.array([[vals[k]]])) for k in range(n)])
    T.tdmrg_set_hamiltonian(ctx, 0, -1, [])
    return ctx, (n - 1, 0), np.repeat(vals, dims)


@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 5000, 152 * 128, 152 * 128 + 1, 400_003, 1_100_000])
@pytest.mark.parametrize("nk", [1, 3, 9])
def test_advance(n, nk):
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(n)
    m = min(nk, n)
    cut = np.sort(rng.choice(np.arange(1, n), m - 1, replace=False)) if m > 1 else np.array([], int)
    dims = np.diff(np.concatenate([[0], cut, [n]])).astype(int)
    ctx, Q, lam = _ctx(T, list(zip(np.linspace(-2, 3, m), dims)))
    try:
        phi = rng.standard_normal(n) + 1j * rng.standard_normal(n)
        times = [0.0, 0.4, 1.0]
        tg = [dev(np.zeros(n)) for _ in times]
        for _ in range(2):   # the second run finds the first one's partial-sum slots emptied
            T.tdmrg_evolve(ctx, Q, dev(phi), times, nk, tg)
        used, _, _, _ = T.tdmrg_evolve_info(ctx)
        assert used <= m
        for t, x in zip(times, tg):
            assert np.abs(host(x) - np.exp(-1j * lam * t) * phi).max() <= nk ** 2 * 2.0 ** -50 * np.linalg.norm(phi)
    finally:
        T.tdmrg_destroy(ctx)


@pytest.mark.parametrize("lens", [[1, 1], [3, 70000, 1, 129], [128] * 40, [200_000, 5, 300_000, 64]])
def test_segments(lens):
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(len(lens))
    n = sum(lens)
    ctx, Q, lam = _ctx(T, [(0.3 * k - 1.0, d) for k, d in enumerate(lens)])
    try:
        phi = rng.standard_normal(n) + 1j * rng.standard_normal(n)
        phi[:lens[0]] = 0.0     # the first segment has no start vector
        times = [0.5, 0.0]
        tg = [dev(np.full(n, np.nan)) for _ in times]
        for _ in range(2):
            T.tdmrg_evolve_segments(ctx, Q, dev(phi), lens, times, 6, tg)
        used, _ = T.tdmrg_evolve_segments_info(ctx, Q, 6, len(lens))
        assert used[0] == 0 and np.all(used[1:] == 1)     # one eigenvalue per segment: breakdown after one vector
        for t, x in zip(times, tg):
            assert np.abs(host(x) - np.exp(-1j * lam * t) * phi).max() <= 36 * 2.0 ** -50 * np.linalg.norm(phi)
    finally:
        T.tdmrg_destroy(ctx)
