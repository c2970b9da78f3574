"""The tensor path's H psi of a direct sum is, to the bit, that of its superblocks alone: the tensor products are exact
sums, and the thin FP64 products (slices up to 4) and the tasks left to the FP64 kernel (5 and 6 slices, sums of
several segments) add in an order that depends on the superblock itself, not on what is launched beside it."""
import pytest

from test_gpu_batch import JOBS
from tests.gpu_util import new_ctx, torch_cuda
from workloads import sectors as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slices", [2, 4, 5, 6])
def test_tensor_hpsi_bits(slices):
    torch = torch_cuda()
    from paper_1103_5391_gb300 import problem
    from paper_1103_5391_gb300 import tdmrg as T
    jobs, big = [], new_ctx(prec=T.TDMRG_OZAKI_BF16, ozaki_slices=slices)
    try:
        for L, m, U, nb, seed in JOBS + [(8, 16, 4.0, 1, 104), (10, 40, 1.0, 1, 105)]:
            ss = S.make_synthetic(L, m, U, nbonds=nb, seed=seed)
            ctx = new_ctx(prec=T.TDMRG_OZAKI_BF16, ozaki_slices=slices)
            problem.load_synthetic(ctx, ss)
            jobs.append((ss, ctx, torch.as_tensor(ss.psi_gs).cuda()))
        Qsum, off = T.tdmrg_direct_sum(big, [c for _, c, _ in jobs], [ss.Q0 for ss, _, _ in jobs])
        x = torch.cat([p for _, _, p in jobs])
        y = torch.zeros_like(x)
        T.tdmrg_apply_h(big, Qsum, x, y)
        for k, (ss, ctx, p) in enumerate(jobs):
            yk = torch.zeros_like(p)
            T.tdmrg_apply_h(ctx, ss.Q0, p, yk)
            assert torch.equal(y[off[k]: off[k + 1]], yk), k
    finally:
        T.tdmrg_destroy(big)
        for _, c, _ in jobs:
            T.tdmrg_destroy(c)

