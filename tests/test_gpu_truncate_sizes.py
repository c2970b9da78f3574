"""The truncation kernel around the number of keys its threads hold (8 x 1024), around what its shared memory holds
(25,600 eigenvalues) and beyond, with planted ties across sectors, negative rounding-size eigenvalues and zeros, against
the rule itself; two sides of one context and a changed block (their sector tables are kept between calls).  Kept
counts are whole numbers; the dropped weight is a sum of n terms: n 2^-53 of their absolute sum."""
import numpy as np
import pytest

from gpu_util import new_ctx
from oracle import dmrg

pytestmark = pytest.mark.gpu


def _spectra(rng, dims):
    out = []
    for d in dims:
        lam = 10.0 ** -rng.uniform(0, 18, d)
        lam[rng.random(d) < 0.1] = 0.25
        lam[rng.random(d) < 0.05] = 0.0
        lam[rng.random(d) < 0.05] *= -1e-12
        out.append(np.sort(lam)[::-1])
    return out


def _truncate(T, ctx, side, evals, m):
    import torch
    kept = torch.full((len(evals),), -1, dtype=torch.int32, device="cuda")
    disc = torch.full((1,), np.nan, dtype=torch.float64, device="cuda")
    T.tdmrg_truncate(ctx, torch.from_numpy(np.concatenate(evals)).cuda(), m, kept, disc, side=side)
    return kept.cpu().numpy().tolist(), disc.item()


def _check(T, ctx, side, evals, m):
    kept, disc = _truncate(T, ctx, side, evals, m)
    assert kept == dmrg.kept_counts(evals, m)
    rest = np.concatenate([e[k:] for e, k in zip(evals, kept)])
    assert abs(disc - rest.sum()) <= len(rest) * 2.0 ** -53 * np.abs(rest).sum() + 1e-300


@pytest.mark.parametrize("total", [5, 1023, 8191, 8193, 25600, 25601, 60000])
def test_sizes(total):
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(total)
    nsec = min(total, 97)
    dims = [total // nsec + (k < total % nsec) for k in range(nsec)]
    ctx = new_ctx()
    try:
        T.tdmrg_set_block(ctx, 0, [(k, 0) for k in range(nsec)], dims)
        T.tdmrg_set_block(ctx, 1, [(0, k) for k in range(3)], [4, 1, 7])
        evals, right = _spectra(rng, dims), _spectra(rng, [4, 1, 7])
        for m in sorted({1, total // 3 + 1, total - 1, total, total + 10}):
            _check(T, ctx, 0, evals, m)
            _check(T, ctx, 1, right, min(m, 11))
        T.tdmrg_set_block(ctx, 0, [(0, 0), (1, 1)], [3, 2])
        _check(T, ctx, 0, _spectra(rng, [3, 2]), 4)
    finally:
        T.tdmrg_destroy(ctx)
