"""The measured cases: the calls of time-step-targeting DMRG on synthetic superblocks, through the C ABI's
binding (paper_1103_5391_gb300.tdmrg).

A superblock is the Gaussian sector model of the benchmark (a renormalised block of l sites keeping m states in
sectors (n_up, n_dn) within 5 of l/2, tensored with one site; both blocks alike), its operators and wave
functions drawn on the device from the seed.  Sizes are those of the repository's configurations: the L=8 chain
(tests), L=16 (the Fig. 2 chain, m = 120 and 200), L=32 m=400 (the benchmark), the 2 x 16 ladder m=800, L=48
m=1000, and the serving mix (m in [128, 512]).

Kinds of case ("op"):
  hpsi     one product H psi (tdmrg_apply_h)
  evolve   one Krylov advance with n_v time targets (tdmrg_evolve)
  gs       restarted Lanczos for the ground state (tdmrg_ground_state)
  rho      the weighted reduced density matrix of the ground state and four targets
  eig      the eigendecomposition of a reduced density matrix with a decaying spectrum (tdmrg_rho_eig)
  cut      rho_R -> its eigendecomposition -> the m-state truncation -> H and c^dag in the kept basis, as a sweep does
  corr     a correlation grid <phi| A_i B_j |psi> over lists of left and right operators
  batch    several jobs side by side on the direct sum of their superblocks (tdmrg_evolve_segments)
  step     one time step: advance, rho_L, its eigendecomposition, two observables

Eigenvectors are determined up to a phase each, so what is compared of them is every product u_{ik} conj(u_{i'k})
of neighbouring rows i, i' (every entry enters, the free phase drops out); of a renormalised operator, whose
entry (i, j) carries the phases of states i and j, every entry's modulus.  A ground state, whose sign is free, is
returned with a positive overlap with the start vector.
"""
import math
import random

import numpy as np
import torch

from paper_1103_5391_gb300 import tdmrg as T

N_V, TAU = 4, 0.05
H, CDAG, CANN, DENS = 0, 10, 30, 50     # operator ids: H, 10 + k = c^dag (left) / c (right), 30 + k = its adjoint, 50 = a density


def listed():
    return [
        # the smallest call: H psi of the L=8 chain's superblock, where launches and latency are all there is
        dict(name="hpsi L8 m16 fp64", op="hpsi", L=8, m=16, bonds=1, slices=0, real=False),
        # the product of the benchmark workload on the tensor path
        dict(name="hpsi L32 m400 s4", op="hpsi", L=32, m=400, bonds=1, slices=4, real=False),
        # an ordinary advance in the library's default precision
        dict(name="evolve L16 m120 fp64", op="evolve", L=16, m=120, bonds=1, slices=0, real=False, nk=12),
        # the benchmark's Krylov advance
        dict(name="evolve L32 m400 s4", op="evolve", L=32, m=400, bonds=1, slices=4, real=False, nk=10),
        # the ground state found at every step of a sweep, with the real operators of the Hubbard chain
        dict(name="gs L16 m200 fp64 real", op="gs", L=16, m=200, bonds=1, slices=0, real=True, nk=32, restarts=3),
        # the density matrix at the largest configuration
        dict(name="rho L48 m1000", op="rho", L=48, m=1000, bonds=1, side=0),
        # the truncation's eigenproblem at the benchmark's size and at the largest
        dict(name="eig L32 m400", op="eig", L=32, m=400, bonds=1),
        dict(name="eig L48 m1000", op="eig", L=48, m=1000, bonds=1),
        # one truncation of a sweep that moves left
        dict(name="cut L16 m200 right", op="cut", L=16, m=200, bonds=1, keep=200),
        # Green's function entries on resident states
        dict(name="corr L32 m400 4x4", op="corr", L=32, m=400, bonds=2, n=4),
        # jobs of the serving mix advanced together
        dict(name="batch 6 jobs s4", op="batch", L=32, m=128, m2=256, jobs=6, bonds=1, slices=4, nk=10),
        # a whole time step on the ladder
        dict(name="step 2x16 m800 s4", op="step", L=32, m=800, bonds=2, slices=4, real=False, nk=10),
    ]


def draw(rng):
    op = rng.choice(["hpsi", "evolve", "gs", "rho", "eig", "cut", "corr", "batch", "step"])
    L = 2 * rng.randint(4, 24)
    most = {"gs": 200, "cut": 400, "corr": 400, "batch": 250, "evolve": 700, "step": 600, "hpsi": 1000, "rho": 1000, "eig": 1000}[op]
    m = int(round(math.exp(rng.uniform(math.log(16), math.log(most)))))
    while max(sectors(L, m)[1]) > 152:       # the largest configuration's largest sector: short chains hold fewer states
        m = int(0.85 * m)
    c = dict(op=op, L=L, m=m, bonds=rng.choice([1, 1, 2]))
    if op in ("hpsi", "evolve", "step"):
        c["slices"] = rng.choice([0, 0, 4, 4, 6]) if m <= 300 else 4
        c["real"] = rng.random() < 0.3
    if op in ("evolve", "batch", "step"):
        c["nk"] = rng.randint(6, 14)
    if op == "gs":
        c.update(slices=0, real=rng.random() < 0.7, nk=rng.choice([16, 24, 32]), restarts=rng.randint(1, 3))
    elif op == "rho":
        c["side"] = rng.randint(0, 1)
    elif op == "cut":
        c["keep"] = max(4, int(m * rng.uniform(0.5, 1.2)))
    elif op == "corr":
        c["n"] = rng.randint(1, 4)
    elif op == "batch":
        c.update(slices=rng.choice([0, 4]), jobs=rng.randint(2, 6), m2=int(m * rng.uniform(1.0, 1.6)) + 1)
    return c


# ---------------------------------------------------------------------------------- the superblock (host tables)
def sectors(L, m):
    """Sector table (sorted quantum numbers, dimensions) of one enlarged block."""
    lb = L // 2 - 1
    c = lb / 2.0
    lo, hi = max(math.ceil(c) - 5, 0), min(math.floor(c) + 5, lb)
    w = {(a, b): math.exp(-((a - c) ** 2 + (b - c) ** 2) / 8.0) for a in range(lo, hi + 1) for b in range(lo, hi + 1)}
    tot, acc = sum(w.values()), {}
    for (a, b), x in w.items():
        d = max(1, round(x / tot * m))
        for q in ((a, b), (a + 1, b), (a, b + 1), (a + 1, b + 1)):
            acc[q] = acc.get(q, 0) + d
    qn = sorted(acc)
    return qn, [acc[q] for q in qn]


def pairs(qn, Q):
    """(left sector, right sector) of superblock sector Q, in order (both blocks have the table qn)."""
    at = {q: k for k, q in enumerate(qn)}
    return [(k, at[Q[0] - q[0], Q[1] - q[1]]) for k, q in enumerate(qn) if (Q[0] - q[0], Q[1] - q[1]) in at]


def targets_of(L):
    return (L // 2, L // 2), (L // 2 + 1, L // 2)


class Model:
    """Operators and states of one superblock on the device, all drawn from the seed."""

    def __init__(self, L, m, bonds, seed, real=False, extra=0):
        self.qn, self.dim = sectors(L, m)
        self.Q0, self.Q1 = targets_of(L)
        self.real, self.bonds = real, bonds
        self.gen = torch.Generator(device="cuda").manual_seed(seed)
        at = {q: k for k, q in enumerate(self.qn)}
        radius = (L // 2) * 3.0
        self.ops = [{}, {}]       # per side: id -> (odd, {(out, in): block})
        for side in (0, 1):
            blocks = {}
            for k, d in enumerate(self.dim):
                x = self.gauss(d, d)
                blocks[k, k] = (x + x.mH) * (radius / (4.0 * math.sqrt(d)))
            self.ops[side][H] = (0, blocks)
            for k in range(max(2 * bonds, extra)):
                s = (1, 0) if k % 2 == 0 else (0, 1)
                s = s if side == 0 else (-s[0], -s[1])      # c^dag on the left, c on the right
                blocks = {}
                for i, q in enumerate(self.qn):
                    o = at.get((q[0] + s[0], q[1] + s[1]))
                    if o is not None:
                        blocks[o, i] = self.gauss(self.dim[o], self.dim[i]) / math.sqrt(self.dim[i])
                self.ops[side][CDAG + k] = (1, blocks)
                self.ops[side][CANN + k] = (1, {(i, o): b.mH.contiguous() for (o, i), b in blocks.items()})
            self.ops[side][DENS] = (0, {(i, i): torch.diag(torch.rand(d, generator=self.gen, device="cuda",
                                        dtype=torch.float64)).to(torch.complex128) for i, d in enumerate(self.dim)})
        self.conns = [c for k in range(2 * bonds) for c in ((CDAG + k, CDAG + k, -1.0), (CANN + k, CANN + k, 1.0))]

    def gauss(self, *shape):
        if self.real:
            return torch.randn(*shape, generator=self.gen, device="cuda", dtype=torch.float64).to(torch.complex128)
        return torch.randn(*shape, generator=self.gen, device="cuda", dtype=torch.complex128)

    def state(self, Q):
        n = sum(self.dim[a] * self.dim[b] for a, b in pairs(self.qn, Q))
        x = torch.randn(n, generator=self.gen, device="cuda", dtype=torch.complex128)
        return x / x.norm()

    def load(self, slices, hamiltonian=True):
        ctx = T.tdmrg_create(device=0, stream=torch.cuda.current_stream().cuda_stream, nk_max=32,
                             prec=T.TDMRG_OZAKI_BF16 if slices else T.TDMRG_FP64, ozaki_slices=slices or 4)
        for side in (0, 1):
            T.tdmrg_set_block(ctx, side, self.qn, self.dim)
            for i, (odd, blocks) in self.ops[side].items():
                data = torch.cat([b.reshape(-1) for b in blocks.values()])
                T.tdmrg_set_op_device(ctx, side, i, odd, [self.qn[o] + self.qn[k] for o, k in blocks], data)
        if hamiltonian:
            T.tdmrg_set_hamiltonian(ctx, H, H, self.conns)
        torch.cuda.synchronize()
        return ctx

    def product(self, terms, Qin, Qout, psi):
        """sum_k c_k (A_k P_L) (x) B_k psi from sector Qin to Qout in plain torch (None = identity)."""
        pin, pout = pairs(self.qn, Qin), pairs(self.qn, Qout)
        blk, off = {}, 0
        for a, b in pin:
            n = self.dim[a] * self.dim[b]
            blk[a] = psi[off:off + n].view(self.dim[a], self.dim[b])
            off += n
        rin = dict(pin)
        out = {a: torch.zeros(self.dim[a], self.dim[b], dtype=torch.complex128, device="cuda") for a, b in pout}
        for opL, opR, c in terms:
            left = self.ops[0][opL][1] if opL is not None else {(a, a): None for a, _ in pin}
            odd, right = self.ops[1][opR] if opR is not None else (0, {(b, b): None for _, b in pin})
            rout = dict(pout)
            for (o, i), A in left.items():
                if i not in blk or o not in rout or (rout[o], rin[i]) not in right:
                    continue
                B = right[rout[o], rin[i]]
                x = blk[i] if B is None else blk[i] @ B.T
                x = x if A is None else A @ x
                out[o] += c * (-1 if odd and sum(self.qn[i]) % 2 else 1) * x
        return torch.cat([out[a].reshape(-1) for a, _ in pout])

    def hpsi(self, Q, psi):
        return self.product([(H, None, 1.0), (None, H, 1.0)] + self.conns, Q, Q, psi)


def hpsi_flops(L, m, bonds, real):
    """Operations of one H psi in sector Q1: per product the cheaper order of its two multiplications."""
    qn, dim = sectors(L, m)
    _, Q = targets_of(L)
    at, f = {q: k for k, q in enumerate(qn)}, 0.0
    for a, b in pairs(qn, Q):
        x, y = dim[a], dim[b]
        f += x * y * (x + y)
        for s in ((1, 0), (0, 1), (-1, 0), (0, -1)):
            o, r = at.get((qn[a][0] + s[0], qn[a][1] + s[1])), at.get((qn[b][0] - s[0], qn[b][1] - s[1]))
            if o is not None and r is not None:
                f += bonds * min(x * y * dim[r] + dim[o] * x * dim[r], dim[o] * x * y + dim[o] * y * dim[r])
    return (4.0 if real else 8.0) * f


def op_entries(L, m):
    """(entries of H on one side, entries of one c^dag) of the block."""
    qn, dim = sectors(L, m)
    at = {q: k for k, q in enumerate(qn)}
    return sum(d * d for d in dim), sum(d * dim[at[q[0] + 1, q[1]]] for q, d in zip(qn, dim) if (q[0] + 1, q[1]) in at)


def size(L, m, Q):
    qn, dim = sectors(L, m)
    return sum(dim[a] * dim[b] for a, b in pairs(qn, Q))


def job_sizes(case):
    """(L, m) of the jobs of a batch: m spread between m and m2."""
    n = case["jobs"]
    return [(max(8, case["L"] - 2 * (k % 3)), round(case["m"] + (case["m2"] - case["m"]) * k / max(1, n - 1))) for k in range(n)]


# ---------------------------------------------------------------------------------- preparation
class State:
    def __init__(self):
        self.ctxs = []

    def __del__(self):
        for c in self.ctxs:
            T.tdmrg_destroy(c)


def zeros(n, dtype=torch.complex128):
    return torch.zeros(n, dtype=dtype, device="cuda")


def neighbours(dim):
    """Packed index of the entry one row below (cyclic) in the same sector and column."""
    idx, off = [], 0
    for d in dim:
        idx.append(off + np.roll(np.arange(d * d), -d))
        off += d * d
    return torch.from_numpy(np.concatenate(idx)).cuda()


def spectrum_rho(M):
    """A density matrix (packed, one block per sector, trace 1) with random eigenvectors and eigenvalues that
    decay over four orders of magnitude in every sector."""
    blocks = []
    for d in M.dim:
        q = torch.linalg.qr(M.gauss(d, d).cpu())[0].cuda()      # small: the host does it as fast
        k = torch.arange(d, device="cuda", dtype=torch.float64)
        lam = d * torch.exp(-9.0 * (k + torch.rand(d, generator=M.gen, device="cuda", dtype=torch.float64)) / d)
        r = (q * lam) @ q.mH
        blocks.append(((r + r.mH) / 2).reshape(-1))
    tot, off = 0.0, 0
    x = torch.cat(blocks)
    for d in M.dim:
        tot, off = tot + x[off:off + d * d].view(d, d).diagonal().real.sum(), off + d * d
    return x / tot


def prepare(case, seed):
    s, op = State(), case["op"]
    s.case = case
    if op == "batch":
        s.models = [Model(L, m, case["bonds"], seed * 16 + k) for k, (L, m) in enumerate(job_sizes(case))]
        src = [M.load(case["slices"]) for M in s.models]
        s.phis = [M.state(M.Q1) for M in s.models]
        s.ctx = T.tdmrg_create(device=0, stream=torch.cuda.current_stream().cuda_stream, nk_max=32,
                               prec=T.TDMRG_OZAKI_BF16 if case["slices"] else T.TDMRG_FP64, ozaki_slices=case["slices"] or 4)
        s.Q, off = T.tdmrg_direct_sum(s.ctx, src, [M.Q1 for M in s.models])
        s.ctxs = [s.ctx]
        for c in src:
            T.tdmrg_destroy(c)
        s.lens = [b - a for a, b in zip(off, off[1:])]
        s.phi = torch.cat(s.phis)
        s.out = [zeros(len(s.phi)) for _ in range(N_V)]
        s.times = [x * TAU / (N_V - 1) for x in range(N_V)]
        return s
    M = s.M = Model(case["L"], case["m"], case["bonds"], seed, case.get("real", False), 2 * case.get("n", 0))
    if op == "eig":
        M.ops = [{}, {}]
    s.ctx = M.load(case.get("slices", 0), op in ("hpsi", "evolve", "gs", "step"))
    s.ctxs = [s.ctx]
    s.times = [x * TAU / (N_V - 1) for x in range(N_V)]
    s.wgs, s.w = T.tdmrg_tst_weights(N_V)
    n1 = size(case["L"], case["m"], M.Q1)
    if op in ("hpsi", "evolve", "step"):
        s.phi = M.state(M.Q1)
        s.out = [zeros(n1) for _ in range(1 if op == "hpsi" else N_V)]
    if op == "gs":
        s.start = M.state(M.Q0)
        s.psi = torch.empty_like(s.start)
    if op in ("rho", "cut"):
        s.states = [(M.Q0, M.state(M.Q0))] + [(M.Q1, M.state(M.Q1)) for _ in range(N_V)]
    if op == "step":
        s.gs = M.state(M.Q0)
        s.obs = zeros(2)
    if op in ("rho", "cut", "step", "eig"):
        nr = sum(d * d for d in M.dim)
        s.rho = spectrum_rho(M) if op == "eig" else zeros(nr)
        s.evals, s.U = zeros(sum(M.dim), torch.float64), zeros(nr)
        s.nb = neighbours(M.dim)
    if op == "cut":
        s.kept, s.disc = zeros(len(M.dim), torch.int32), zeros(1, torch.float64)
        s.ren = [zeros(sum(b.numel() for b in M.ops[1][i][1].values())) for i in (H, CDAG, CDAG + 1)]
    if op == "corr":
        s.phi1, s.phi2 = M.state(M.Q0), M.state(M.Q0)
        s.grid = zeros(case["n"] ** 2)
    return s


# ---------------------------------------------------------------------------------- one pass
def run(s):
    case, op = s.case, s.case["op"]
    if op == "batch":
        T.tdmrg_evolve_segments(s.ctx, s.Q, s.phi, s.lens, s.times, case["nk"], s.out)
        return s.out
    M, ctx = s.M, s.ctx
    if op == "hpsi":
        T.tdmrg_apply_h(ctx, M.Q1, s.phi, s.out[0])
        return s.out
    if op == "evolve":
        T.tdmrg_evolve(ctx, M.Q1, s.phi, s.times, case["nk"], s.out)
        return s.out
    if op == "gs":
        s.psi.copy_(s.start)
        e = T.tdmrg_ground_state(ctx, M.Q0, s.psi, case["nk"], case["restarts"])
        return {"energy": e, "psi": s.psi * torch.sgn(torch.vdot(s.psi, s.start))}
    if op == "rho":
        T.tdmrg_density_matrix(ctx, s.states, [s.wgs] + s.w, s.rho, side=case["side"])
        return s.rho
    if op == "eig":
        T.tdmrg_rho_eig(ctx, s.rho, s.evals, s.U)
        return {"evals": s.evals, "vectors": s.U * s.U[s.nb].conj()}
    if op == "cut":
        T.tdmrg_density_matrix(ctx, s.states, [s.wgs] + s.w, s.rho, side=1)
        T.tdmrg_rho_eig(ctx, s.rho, s.evals, s.U, side=1)
        T.tdmrg_truncate(ctx, s.evals, case["keep"], s.kept, s.disc, side=1)
        kept = s.kept.cpu().numpy()
        for i, o in zip((H, CDAG, CDAG + 1), s.ren):
            T.tdmrg_renormalize_op(ctx, 1, i, s.U, kept, o)
        return {"rho": s.rho, "evals": s.evals, "vectors": s.U * s.U[s.nb].conj(), "kept": s.kept, "discarded": s.disc,
                "operators": [o.abs() for o in s.ren]}
    if op == "corr":
        T.tdmrg_correlation(ctx, *corr_ops(case), M.Q0, s.phi1, M.Q0, s.phi2, s.grid)
        return s.grid
    if op == "step":
        T.tdmrg_evolve(ctx, M.Q1, s.phi, s.times, case["nk"], s.out)
        T.tdmrg_density_matrix(ctx, [(M.Q0, s.gs)] + [(M.Q1, x) for x in s.out], [s.wgs] + s.w, s.rho)
        T.tdmrg_rho_eig(ctx, s.rho, s.evals, s.U)
        T.tdmrg_expect(ctx, DENS, -1, M.Q1, s.out[-1], s.obs[0:1])
        T.tdmrg_expect(ctx, -1, DENS, M.Q1, s.out[-1], s.obs[1:2])
        return {"targets": s.out, "rho": s.rho, "evals": s.evals, "vectors": s.U * s.U[s.nb].conj(), "observables": s.obs}
    raise ValueError(op)


def corr_ops(case):
    """c^dag_up of n left sites, c_up of n right sites."""
    ids = [CDAG + 2 * k for k in range(case["n"])]
    return ids, ids


# ---------------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    op = case["op"]
    if op == "batch":
        w = [work(dict(case, op="evolve", L=L, m=m, real=False)) for L, m in job_sizes(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    L, m, real = case["L"], case["m"], case.get("real", False)
    qn, dim = sectors(L, m)
    Q0, Q1 = targets_of(L)
    n0, n1 = size(L, m, Q0), size(L, m, Q1)
    nh, nc = op_entries(L, m)
    ham = 16.0 * (2 * nh + 2 * 4 * case["bonds"] * nc)      # every operator of H read once
    nr = sum(d * d for d in dim)
    if op == "hpsi":
        return {"bytes": ham + 32.0 * n1, "flops": hpsi_flops(L, m, case["bonds"], real)}
    advance = lambda n, nk, out: (ham + 16.0 * n * (1 + out), nk * hpsi_flops(L, m, case["bonds"], real)
                                  + 8.0 * n * nk * (nk + 1) + 8.0 * n * nk * out)
    # rho: the lower triangles of sum_l Psi_l Psi_l^dag
    rho = (16.0 * (n0 + N_V * n1) + 16.0 * nr,
           4.0 * sum(dim[a] ** 2 * dim[b] for a, b in pairs(qn, Q0)) + 4.0 * N_V * sum(dim[a] ** 2 * dim[b] for a, b in pairs(qn, Q1)))
    # a dense Hermitian eigenproblem: reduction, eigenvectors, back transformation
    eig = (32.0 * nr + 8.0 * sum(dim), 24.0 * sum(d ** 3 for d in dim))
    if op == "evolve":
        b, f = advance(n1, case["nk"], N_V)
        return {"bytes": b, "flops": f}
    if op == "gs":
        b, f = advance(n0, case["nk"], 1)
        return {"bytes": b * case["restarts"], "flops": f * case["restarts"]}
    if op == "rho":
        return {"bytes": rho[0], "flops": rho[1]}
    if op == "eig":
        return {"bytes": eig[0], "flops": eig[1]}
    if op == "cut":
        ren = 16.0 * 2 * (nh + 2 * nc)
        return {"bytes": rho[0] + eig[0] + ren, "flops": rho[1] + eig[1] + 16.0 * sum(d ** 3 for d in dim)}
    if op == "corr":
        n, at, f = case["n"], {q: k for k, q in enumerate(qn)}, 0.0
        for a, b in pairs(qn, Q0):
            o, r = at.get((qn[a][0] + 1, qn[a][1])), at.get((qn[b][0] - 1, qn[b][1]))
            if o is not None and r is not None:
                f += 8.0 * n * dim[a] * dim[r] * (dim[b] + n * dim[o])
        return {"bytes": 16.0 * (2 * n0 + 2 * n * nc), "flops": f}
    b, f = advance(n1, case["nk"], N_V)
    return {"bytes": b + rho[0] + eig[0], "flops": f + rho[1] + eig[1]}


# ---------------------------------------------------------------------------------- plain torch in 64 bits
def lanczos(hpsi, v, nk):
    V, al, be = [v / v.norm()], [], []
    for j in range(nk):
        w = hpsi(V[-1])
        al.append(torch.vdot(V[-1], w).real.item())
        B = torch.stack(V)
        for _ in range(2):
            w = w - B.T @ (B.conj() @ w)
        if j + 1 < nk:
            be.append(w.norm().item())
            V.append(w / be[-1])
    return torch.stack(V), np.diag(al) + np.diag(be, 1) + np.diag(be, -1)


def advance_exact(M, phi, times, nk):
    V, t = lanczos(lambda v: M.hpsi(M.Q1, v), phi, nk)
    w, S = np.linalg.eigh(t)
    c = [S @ (np.exp(-1j * w * x) * S[0]) * phi.norm().item() for x in times]
    return [V.T @ torch.from_numpy(x).cuda() for x in c]


def rho_exact(M, states, weights, side):
    out = [torch.zeros(d, d, dtype=torch.complex128, device="cuda") for d in M.dim]
    for (Q, psi), w in zip(states, weights):
        off, w = 0, w / torch.vdot(psi, psi).real
        for a, b in pairs(M.qn, Q):
            n = M.dim[a] * M.dim[b]
            x = psi[off:off + n].view(M.dim[a], M.dim[b])
            off += n
            if side == 0:
                out[a] += w * (x @ x.mH)
            else:
                out[b] += w * (x.T @ x.conj())
    return torch.cat([r.reshape(-1) for r in out])


def eig_exact(M, rho, nb):
    rho, ev, U, off = rho.cpu(), [], [], 0
    for d in M.dim:
        w, u = torch.linalg.eigh(rho[off:off + d * d].view(d, d))
        ev.append(w.flip(0))
        U.append(u.flip(1))
        off += d * d
    flat = torch.cat([u.reshape(-1) for u in U]).cuda()
    return torch.cat(ev).cuda(), flat * flat[nb].conj(), U


def exact(case, seed):
    s, op = prepare(case, seed), case["op"]
    if op == "batch":
        per = [advance_exact(M, p, s.times, case["nk"]) for M, p in zip(s.models, s.phis)]
        return [torch.cat([x[k] for x in per]) for k in range(N_V)]
    M = s.M
    if op == "hpsi":
        return [M.hpsi(M.Q1, s.phi)]
    if op == "evolve":
        return advance_exact(M, s.phi, s.times, case["nk"])
    if op == "gs":
        v = s.start
        for _ in range(case["restarts"]):
            V, t = lanczos(lambda x: M.hpsi(M.Q0, x), v, case["nk"])
            w, S = np.linalg.eigh(t)
            v = V.T @ torch.from_numpy(S[:, 0]).cuda().to(torch.complex128)
        return {"energy": float(w[0]), "psi": v * torch.sgn(torch.vdot(v, s.start))}
    if op == "rho":
        return rho_exact(M, s.states, [s.wgs] + s.w, case["side"])
    if op == "eig":
        ev, vec, _ = eig_exact(M, s.rho, s.nb)
        return {"evals": ev, "vectors": vec}
    if op == "cut":
        rho = rho_exact(M, s.states, [s.wgs] + s.w, 1)
        ev, vec, U = eig_exact(M, rho, s.nb)
        order = torch.sort(ev, descending=True).indices[:case["keep"]].cpu().tolist()
        bound = np.cumsum(M.dim)
        kept = [0] * len(M.dim)
        for i in order:
            kept[int(np.searchsorted(bound, i, side="right"))] += 1
        rest = [x for k, w in enumerate(torch.split(ev.cpu(), M.dim)) for x in w[kept[k]:].tolist()]
        ops = []
        for i, o in zip((H, CDAG, CDAG + 1), s.ren):
            full, off = torch.zeros(len(o), dtype=torch.float64, device="cuda"), 0
            for (a, b), x in M.ops[1][i][1].items():
                y = (U[a][:, :kept[a]].cuda().mH @ x @ U[b][:, :kept[b]].cuda()).abs().reshape(-1)
                full[off:off + len(y)] = y
                off += len(y)
            ops.append(full)
        return {"rho": rho, "evals": ev, "vectors": vec, "kept": torch.tensor(kept, dtype=torch.int32),
                "discarded": torch.tensor([math.fsum(rest)], dtype=torch.float64), "operators": ops}
    if op == "corr":
        a, b = corr_ops(case)
        return torch.stack([torch.vdot(s.phi1, M.product([(i, j, 1.0)], M.Q0, M.Q0, s.phi2)) for i in a for j in b])
    tg = advance_exact(M, s.phi, s.times, case["nk"])
    rho = rho_exact(M, [(M.Q0, s.gs)] + [(M.Q1, x) for x in tg], [s.wgs] + s.w, 0)
    ev, vec, _ = eig_exact(M, rho, s.nb)
    x = tg[-1]
    obs = [torch.vdot(x, M.product([t], M.Q1, M.Q1, x)) / torch.vdot(x, x).real for t in ((DENS, None, 1.0), (None, DENS, 1.0))]
    return {"targets": tg, "rho": rho, "evals": ev, "vectors": vec, "observables": torch.stack(obs)}
