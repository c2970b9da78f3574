"""The first call of every kind on a context that runs on a non-blocking stream, while the default stream still has work
queued: the tables that the call builds are in place before its kernels read them, so the results are, to the bit, those
of a context whose default stream was idle."""
import numpy as np
import pytest

from gpu_util import torch_cuda
from workloads import sectors as S

pytestmark = pytest.mark.gpu


def _results(T, problem, ss, prec, stream, busy):
    """Outputs of the first calls on a fresh context; busy() queues work on the default stream before each of them."""
    import torch
    ctx = T.tdmrg_create(device=torch.cuda.current_device(), stream=stream.cuda_stream, prec=prec, ozaki_slices=4, nk_max=32)
    out = []
    try:
        problem.load_synthetic(ctx, ss)
        psi = torch.as_tensor(ss.psi_gs).cuda()
        n1 = T.tdmrg_sector_size(ctx, ss.Q1)
        y, phi = torch.zeros_like(psi), torch.zeros(n1, dtype=torch.complex128, device="cuda")
        tg = [torch.zeros_like(phi) for _ in range(3)]
        gs = psi.clone()
        nr, ne = T.tdmrg_rho_size(ctx)
        rho, U = (torch.zeros(nr, dtype=torch.complex128, device="cuda") for _ in range(2))
        ev = torch.zeros(ne, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        for call in (lambda: T.tdmrg_apply_h(ctx, ss.Q0, psi, y),
                     lambda: T.tdmrg_apply_op(ctx, -1, problem.OP_EXC, ss.Q0, psi, ss.Q1, phi),
                     lambda: T.tdmrg_evolve(ctx, ss.Q1, phi, [0.0, 0.05, 0.1], 8, tg),
                     lambda: T.tdmrg_ground_state(ctx, ss.Q0, gs, nk=6, restarts=1),
                     lambda: T.tdmrg_density_matrix(ctx, [(ss.Q0, psi), (ss.Q1, phi)], [0.5, 0.5], rho),
                     lambda: T.tdmrg_rho_eig(ctx, rho, ev, U)):
            busy()
            call()
        torch.cuda.synchronize()
        out = [t.cpu() for t in (y, phi, *tg, gs, rho, ev, U)]
    finally:
        T.tdmrg_destroy(ctx)
    return out


@pytest.mark.parametrize("tensor", [False, True])
def test_first_calls_beside_default_stream_work(tensor):
    torch = torch_cuda()
    from paper_1103_5391_gb300 import problem
    from paper_1103_5391_gb300 import tdmrg as T
    prec = T.TDMRG_OZAKI_BF16 if tensor else T.TDMRG_FP64
    ss = S.make_synthetic(16, 96, 4.0, nbonds=1, seed=11)
    stream = torch.cuda.Stream()
    x = torch.zeros(1 << 26, device="cuda")

    def busy():
        with torch.cuda.stream(torch.cuda.default_stream()):
            for _ in range(40):
                x.add_(1.0)

    idle = _results(T, problem, ss, prec, stream, lambda: None)
    for got, want in zip(_results(T, problem, ss, prec, stream, busy), idle):
        assert torch.equal(got, want)
    assert np.isfinite(float(x[0]))
