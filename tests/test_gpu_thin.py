"""The thin products of the tensor kernel: outputs around 32 (a warp), several tasks in one warp, outputs shared by up to
eight lanes (segments and parts of K), real and complex operands and factors, both store orders.

Every product of these sizes is thin (at most 8 steps of four k over its segments), so H psi with four slices has FP64's
error: an output is a sum of products of T = K_1 + K_2 terms in all its segments, each complex multiply-add with at most
4 roundings and each sum over lanes with at most 3 more, so |error| <= 4 (T + 8) 2^-53 sum |a| |b| |c|, element by element.
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
    (1, 1, 0, False), (1, 31, 1, False), (1, 32, 2, True), (3, 11, 1, False), (11, 3, 1, True), (2, 17, 6, False),
    (4, 8, 5, False), (5, 5, 2, True), (32, 1, 0, False), (31, 32, 0, False), (8, 4, 2, False), (16, 16, 0, True)])
def test_thin_product(dl, dr, nconn, real):
    from paper_1103_5391_gb300 import tdmrg as T
    rng = np.random.default_rng(dl * 1000 + dr)
    HL, HR = _rand(rng, real, dl, dl), _rand(rng, real, dr, dr)
    A = [_rand(rng, real, dl, dl) for _ in range(nconn)]
    B = [_rand(rng, False if k % 3 == 1 else real, dr, dr) for k in range(nconn)]
    co = [complex(0.5 + k, 0.0 if k % 2 == 0 else -1.25) for k in range(nconn)]
    psi = _rand(rng, False, dl, dr)
    ctx = new_ctx(prec=T.TDMRG_OZAKI_BF16, ozaki_slices=4)
    try:
        T.tdmrg_set_thin_dim(ctx, 64)
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
