"""The factorised correlation grid against the entries taken one by one (tdmrg_overlap_op): identities on either side,
lists whose operators shift the sector differently (products that do not lead to phi1's sector give zero), real and
complex operators, different sectors of the two states, repeated calls on one plan.  Both sides are FP64 sums of
the same products in another order; with unit states and operators of norm below 100 an entry is bounded by
100^2 times (terms 2^-50), 1e-9 at these sizes."""
import numpy as np
import pytest

from gpu_util import dev, host, new_ctx
from workloads import sectors as S

pytestmark = pytest.mark.gpu

CASES = {
    "green": ([10, 12], [10, 12], 0, 0),
    "identities left": ([-1, 50, 0], [50, 0], 0, 0),
    "identities right": ([50, 0], [-1, 50], 1, 1),
    "one by one": ([50], [50], 1, 1),
    "mixed shifts": ([10, 50, 11, 0], [50, 10, 11], 0, 0),
    "between sectors": ([-1], [49], 1, 0),
    "left shift only": ([10, 11], [-1], 1, 0),
    "nothing connects": ([10], [30], 0, 1),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("real", [False, True])
def test_grid_equals_entries(name, real):
    from paper_1103_5391_gb300 import problem
    from paper_1103_5391_gb300 import tdmrg as T
    left, right, k1, k2 = CASES[name]
    ss = S.make_synthetic(12, 40, 4.0, nbonds=2, seed=S.SEED_BASE + 3)
    if real:
        for ops in [ss.HL, ss.HR, ss.cdag_exc] + [x for b in ss.cdagL + ss.cR for x in b]:
            for k in ops:
                ops[k] = ops[k].real + 0j
    Qs = (ss.Q0, ss.Q1)
    rng = np.random.default_rng(4)
    ctx = new_ctx()
    try:
        problem.load_synthetic(ctx, ss)
        state = lambda Q: (lambda v: v / np.linalg.norm(v))(rng.standard_normal(ss.sector_size(Q)) + 1j * rng.standard_normal(ss.sector_size(Q)))
        for _ in range(2):
            phi1, phi2 = dev(state(Qs[k1])), dev(state(Qs[k2]))
            out = dev(np.full(len(left) * len(right), np.nan))
            T.tdmrg_correlation(ctx, left, right, Qs[k1], phi1, Qs[k2], phi2, out)
            got = host(out).reshape(len(left), len(right))
            one = dev(np.zeros(1))
            for i, a in enumerate(left):
                for j, b in enumerate(right):
                    if a < 0 and b < 0:
                        continue
                    T.tdmrg_overlap_op(ctx, a, b, Qs[k1], phi1, Qs[k2], phi2, one)
                    assert abs(got[i, j] - host(one)[0]) <= 1e-9
    finally:
        T.tdmrg_destroy(ctx)
