"""The grouped FP64 GEMM at the edges of its tiles: outputs around 32 and 256 (lanes, a tile), K from 1 up,
more segments than one tile takes, real and complex operands and factors, Hermitian results of odd sizes.

Bound: an output is a sum of products of T = K_1 + K_2 terms in all its segments (two chained products for a
connection), each complex multiply-add with at most 4 roundings, so |error| <= 4 (T + 8) 2^-53 sum |a| |b| |c|,
element by element.
"""
import numpy as np
import pytest

from gpu_util import dev, host, new_ctx

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


def _rand(rng, real, *shape):
    x = rng.standard_normal(shape)
    return x.astype(complex) if real else x + 1j * rng.standard_normal(shape)


@pytest.mark.parametrize("dl,dr,nconn,real", [
    (1, 1, 0, False), (1, 31, 1, False), (4, 8, 2, True), (3, 11, 1, False), (51, 5, 3, False), (16, 16, 1, True),
    (257, 1, 0, False), (1, 257, 2, False), (13, 20, 17, False), (7, 9, 60, False), (90, 131, 2, False), (200, 60, 1, True)])
def test_product(dl, dr, nconn, real):
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(dl * 1000 + dr)
    HL, HR = _rand(rng, real, dl, dl), _rand(rng, real, dr, dr)
    A = [_rand(rng, real, dl, dl) for _ in range(nconn)]
    B = [_rand(rng, False if k % 3 == 1 else real, dr, dr) for k in range(nconn)]
    co = [complex(0.5 + k, 0.0 if k % 2 == 0 else -1.25) for k in range(nconn)]
    psi = _rand(rng, False, dl, dr)
    ctx = new_ctx()
    try:
        T.tdmrg_set_block(ctx, 0, [(0, 0)], [dl])
        T.tdmrg_set_block(ctx, 1, [(0, 0)], [dr])
        one = lambda x: [((0, 0), (0, 0), x)]
        T.tdmrg_set_op(ctx, 0, 0, 0, one(HL))
        T.tdmrg_set_op(ctx, 1, 0, 0, one(HR))
        for k in range(nconn):
            T.tdmrg_set_op(ctx, 0, 1 + k, 0, one(A[k]))
            T.tdmrg_set_op(ctx, 1, 1 + k, 0, one(B[k]))
        T.tdmrg_set_hamiltonian(ctx, 0, 0, [(1 + k, 1 + k, co[k]) for k in range(nconn)])
        out = dev(np.full(dl * dr, np.nan))
        for _ in range(2):   # a second product finds the split-K tickets at zero again
            T.tdmrg_apply_h(ctx, (0, 0), dev(psi.reshape(-1)), out)
        got = host(out).reshape(dl, dr)
    finally:
        T.tdmrg_destroy(ctx)
    want = HL @ psi + psi @ HR.T + sum(c * (a @ psi @ b.T) for c, a, b in zip(co, A, B))
    aps = np.abs(psi)
    mag = np.abs(HL) @ aps + aps @ np.abs(HR).T + sum((abs(c) * (np.abs(a) @ aps @ np.abs(b).T) for c, a, b in zip(co, A, B)),
                                                      np.zeros((dl, dr)))
    terms = (nconn + 1) * (dl + dr)
    assert np.all(np.abs(got - want) <= 2 * 4 * (terms + 8) * EPS * mag)   # numpy's own roundings: the factor 2


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("dims,nt", [([1], 1), ([7, 8], 3), ([22, 23, 31], 2), ([33, 3, 100], 12), ([150, 1], 5)])
def test_hermitian(dims, nt, side):
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(sum(dims) + nt)
    n = len(dims)
    other = [d + 2 * k + 1 for k, d in enumerate(dims)][::-1]
    qn = [(k, 0) for k in range(n)]
    Q = (n - 1, 0)
    ld, rd = (dims, other) if side == 0 else (other, dims)
    psis = [[_rand(rng, False, ld[k], rd[n - 1 - k]) for k in range(n)] for _ in range(nt)]
    w = (0.1 + rng.random(nt)).tolist()
    ctx = new_ctx()
    try:
        T.tdmrg_set_block(ctx, 0, qn, ld)
        T.tdmrg_set_block(ctx, 1, qn, rd)
        rho = dev(np.full(sum(d * d for d in dims), np.nan))
        for _ in range(2):
            T.tdmrg_density_matrix(ctx, [(Q, dev(np.concatenate([x.reshape(-1) for x in p]))) for p in psis], w, rho, side=side)
        got = host(rho)
    finally:
        T.tdmrg_destroy(ctx)
    off = 0
    for k, d in enumerate(dims):
        r = got[off:off + d * d].reshape(d, d)
        off += d * d
        want, mag, terms = np.zeros((d, d), complex), np.zeros((d, d)), 0
        for p, wl in zip(psis, w):
            x = p[k] if side == 0 else p[n - 1 - k].T
            f = wl / sum(np.sum(np.abs(y) ** 2) for y in p)
            want += f * (x @ x.conj().T)
            mag += f * (np.abs(x) @ np.abs(x).T)
            terms += x.shape[1]
        # the norms: sums of positive terms, relative error below (length of the vector) 2^-53
        terms += sum(y.size for y in psis[0])
        assert np.all(np.abs(r - want) <= 2 * 4 * (terms + 8) * EPS * mag)
        assert np.array_equal(r, r.conj().T)
