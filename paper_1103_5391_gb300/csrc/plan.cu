// Sector bookkeeping: compiles a superblock product sum_k coeff_k (A_k P_L^{odd B_k}) (x) B_k from
// sector Q_in to Q_out into two grouped lists of small complex GEMMs (Sec. IV, the "Hamiltonian
// connections" between the two blocks; superblock sectors of Sec. II.B).
//
// For an input pair (q', r' = Q_in - q') and a term with blocks A[q <- q'] and B[r <- r'] such that
// (q, r) is a pair of Q_out, the contribution is
//     Psi'_q += coeff * s(q') * A Psi_{q'} B^T,     s(q') = (-1)^{N(q')} if B is odd, else 1.
// Stage 1 (right products):   T = Psi_{q'} B^T  into scratch, or straight into Psi'_q when A = 1;
// stage 2 (left products):    Psi'_q = [stage-1 value] + sum coeff s A T  (and A Psi_{q'} when B = 1).
// Each stage-2 output block owns one task whose segments are all its left products, so every
// output tile accumulates all of its terms in registers before a single store (no atomics).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "internal.h"

namespace tdmrg {

int upload(tdmrg_ctx* c, TaskList& tl) {   // uploads_done follows, once for all lists of a build
    release(c, tl);
    struct { void** dst; const void* src; size_t bytes; } parts[4] = {
        {(void**)&tl.d_tasks, tl.tasks.data(), tl.tasks.size() * sizeof(Task)},
        {(void**)&tl.d_segs, tl.segs.data(), tl.segs.size() * sizeof(Seg)},
        {(void**)&tl.d_tiles, tl.tiles.data(), tl.tiles.size() * sizeof(Tile)},
        {(void**)&tl.d_ctiles, tl.ctiles.data(), tl.ctiles.size() * sizeof(CorrTile)}};
    for (auto& pt : parts) {
        if (!pt.bytes) continue;
        int rc = dev_alloc(c, pt.dst, pt.bytes, "task list");
        if (rc) return rc;
        // synchronous copy: the host vectors may be rebuilt before the stream reaches this point
        rc = cuda_check(c, cudaMemcpy(*pt.dst, pt.src, pt.bytes, cudaMemcpyHostToDevice), "task list upload");
        if (rc) return rc;
    }
    if (tl.nsplit) {
        int rc = dev_alloc(c, (void**)&tl.d_partials, (size_t)tl.npartial * sizeof(cplx),
                           "split-K partials");
        if (!rc) rc = dev_alloc(c, (void**)&tl.d_counters, (size_t)tl.nsplit * sizeof(int), "split-K tickets");
        if (!rc) rc = cuda_check(c, cudaMemset(tl.d_counters, 0, (size_t)tl.nsplit * sizeof(int)), "split-K tickets");
        if (rc) return rc;
    }
    tl.bytes = tl.tasks.size() * sizeof(Task) + tl.segs.size() * sizeof(Seg) + tl.tiles.size() * sizeof(Tile) +
               tl.ctiles.size() * sizeof(CorrTile) +
               (size_t)tl.npartial * sizeof(cplx) + (size_t)tl.nsplit * sizeof(int);
    return TDMRG_OK;
}

void release(tdmrg_ctx* c, TaskList& tl) {
    if (tl.d_tasks) dev_free(c, tl.d_tasks, tl.tasks.size() * sizeof(Task));
    if (tl.d_segs) dev_free(c, tl.d_segs, tl.segs.size() * sizeof(Seg));
    if (tl.d_tiles) dev_free(c, tl.d_tiles, tl.tiles.size() * sizeof(Tile));
    if (tl.d_ctiles) dev_free(c, tl.d_ctiles, tl.ctiles.size() * sizeof(CorrTile));
    if (tl.d_partials) dev_free(c, tl.d_partials, (size_t)tl.npartial * sizeof(cplx));
    if (tl.d_counters) dev_free(c, tl.d_counters, (size_t)tl.nsplit * sizeof(int));
    tl.d_tasks = nullptr; tl.d_segs = nullptr; tl.d_tiles = nullptr; tl.d_ctiles = nullptr; tl.d_partials = nullptr; tl.d_counters = nullptr;
}

int run_transient(tdmrg_ctx* c, TaskList* const* lists, int nlists, int64_t scratch, GemmArgs g, const char* what) {
    // one device buffer: scratch | per list: tasks, segments, tiles | tickets | partial sums.  It stays with the context
    // (grown when a call needs more), so that a call costs one copy and no allocation; dev_alloc gives it back
    // when memory runs out.  One copy per call from a host image of the tables and zeroed tickets.
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    struct Off { size_t tasks, segs, tiles, tick, part; };
    std::vector<Off> off(nlists);
    const size_t b_scr = al((size_t)scratch * sizeof(cplx));
    size_t pos = b_scr;
    for (int k = 0; k < nlists; ++k) {
        off[k].tasks = pos; pos += al(lists[k]->tasks.size() * sizeof(Task));
        off[k].segs = pos; pos += al(lists[k]->segs.size() * sizeof(Seg));
        off[k].tiles = pos; pos += al(lists[k]->tiles.size() * sizeof(Tile));
        off[k].tick = pos; pos += al((size_t)lists[k]->nsplit * sizeof(int));
    }
    const size_t b_tab = pos - b_scr;
    for (int k = 0; k < nlists; ++k) { off[k].part = pos; pos += al((size_t)lists[k]->npartial * sizeof(cplx)); }
    if (c->transient_bytes < pos) {
        dev_free(c, c->transient, c->transient_bytes);
        c->transient = nullptr;
        c->transient_bytes = 0;
        int rc = dev_alloc(c, &c->transient, pos, what);
        if (rc) return rc;
        c->transient_bytes = pos;
    }
    unsigned char* base = static_cast<unsigned char*>(c->transient);
    std::vector<unsigned char> host(b_tab, 0);
    for (int k = 0; k < nlists; ++k) {
        const TaskList& tl = *lists[k];
        if (!tl.tasks.empty()) memcpy(host.data() + off[k].tasks - b_scr, tl.tasks.data(), tl.tasks.size() * sizeof(Task));
        if (!tl.segs.empty()) memcpy(host.data() + off[k].segs - b_scr, tl.segs.data(), tl.segs.size() * sizeof(Seg));
        if (!tl.tiles.empty()) memcpy(host.data() + off[k].tiles - b_scr, tl.tiles.data(), tl.tiles.size() * sizeof(Tile));
    }
    int rc = b_tab ? cuda_check(c, cudaMemcpyAsync(base + b_scr, host.data(), b_tab, cudaMemcpyHostToDevice, c->stream), what) : TDMRG_OK;
    g.bufs[BUF_SCRATCH] = reinterpret_cast<cplx*>(base);
    for (int k = 0; k < nlists && !rc; ++k) {
        if (lists[k]->tiles.empty()) continue;
        g.tasks = reinterpret_cast<const Task*>(base + off[k].tasks);
        g.segs = reinterpret_cast<const Seg*>(base + off[k].segs);
        g.tiles = reinterpret_cast<const Tile*>(base + off[k].tiles);
        g.ntiles = (int)lists[k]->tiles.size();
        g.counters = reinterpret_cast<int*>(base + off[k].tick);
        g.partials = reinterpret_cast<cplx*>(base + off[k].part);
        c->launches++;
        rc = cuda_check(c, launch_gemm_f64(g, c->stream, nullptr, 0), what);
    }
    // the products are done before the buffer and the host image are used again
    const int rc2 = cuda_check(c, cudaStreamSynchronize(c->stream), what);
    return rc ? rc : rc2;
}

int64_t sector_size(const tdmrg_ctx* c, int n_up, int n_dn) {
    const Side& L = c->side[0];
    const Side& R = c->side[1];
    int64_t n = 0;
    for (size_t qi = 0; qi < L.dim.size(); ++qi) {
        int ri = R.find(n_up - L.nup[qi], n_dn - L.ndn[qi]);
        if (ri >= 0) n += (int64_t)L.dim[qi] * R.dim[ri];
    }
    return n;
}

// Tiles of the grouped FP64 GEMM.  The K range one warp runs through aims at half the launch's work per FP64 pipe
// (152 SMs x 4), between 8 and 192: small launches are cut finely so that every pipe has work and no chain is long,
// but not more finely than that needs, as a CTA's fixed latency (its tables, the first operands, the sums of its
// shares: ~6000 cycles) is that of ~25 complex k of a warp.  Measured: a sixth of the work instead of half makes a ground
// state at L=16 m=200 25 % slower, a floor of 4 or 16 instead of 8 a Krylov advance at L=16 m=120 17 % or 3 %, a cap of 64
// instead of 192 rho_L at L=48 m=1000 4 %.
// With groups (group[t] of task t) the work is that of the task's group alone, so that the sums of a group's outputs do
// not depend on what else is launched with it.
// A task's K is divided first among the warps of a CTA (ks = 1, 2, 4, 8 shares, 256 / ks outputs), then over CTAs.
void make_tiles(TaskList& tl, const std::vector<int>* group) {
    tl.tiles.clear();
    tl.flops = 0.0;
    tl.nsplit = 0;
    tl.npartial = 0;
    std::vector<double> work(1, 0.0);
    std::vector<int64_t> outs(tl.tasks.size()), ks(tl.tasks.size(), 0);
    for (size_t t = 0; t < tl.tasks.size(); ++t) {
        const Task& k = tl.tasks[t];
        outs[t] = k.herm ? (int64_t)k.M * (k.M + 1) / 2 : (int64_t)k.M * k.N;
        for (int s = k.seg_begin; s < k.seg_end; ++s) {
            ks[t] += tl.segs[s].K;
            // 8 real flops per complex multiply-add, 4 when one operand is real
            tl.flops += (tl.segs[s].rflags ? 4.0 : 8.0) * (double)k.M * k.N * (double)tl.segs[s].K;
        }
        const size_t gr = group ? (size_t)(*group)[t] : 0;
        if (gr >= work.size()) work.resize(gr + 1, 0.0);
        work[gr] += (double)outs[t] * (double)ks[t];
    }
    for (size_t t = 0; t < tl.tasks.size(); ++t) {
        const Task& k = tl.tasks[t];
        if (outs[t] <= 0) continue;
        const int64_t per_warp = (int64_t)std::min(192.0, std::max(8.0, work[group ? (*group)[t] : 0] / (32.0 * 608.0 * 2.0)));
        const int64_t shares = std::max<int64_t>(1, (ks[t] + per_warp - 1) / per_warp);
        const int cks = shares <= 1 ? 1 : shares <= 2 ? 2 : shares <= 4 ? 4 : 8;
        const int area = kTileOut / cks;
        int want = (int)std::min<int64_t>({(shares + cks - 1) / cks, (int64_t)kMaxParts, std::max<int64_t>(ks[t], 1)});
        // sector products: parts of 96 k and a segment at least (a tile's segments may ask for more), so that the partial
        // sums stay within what the allocation-free product's static array is made for: one part per 96 k (a Krylov
        // advance at L=16 m=120 is 1 % faster for it).
        if (group) want = (int)std::min<int64_t>({(int64_t)want, (ks[t] + 95) / 96, std::max<int64_t>(k.seg_end - k.seg_begin, 1)});
        want = std::max(want, 1);
        // K parts [lo, hi) of the concatenated range, each within kTileSegs segments
        struct Part { int seg_lo, seg_hi; int64_t k0, k1; };
        std::vector<Part> parts;
        for (;; ++want) {
            parts.clear();
            bool ok = true;
            for (int p = 0; p < want; ++p) {
                const int64_t lo = ks[t] * p / want, hi = ks[t] * (p + 1) / want;
                int s0 = k.seg_begin;
                int64_t pos = 0;
                while (s0 < k.seg_end && pos + tl.segs[s0].K <= lo) pos += tl.segs[s0++].K;
                int s1 = s0;
                int64_t end = pos;
                while (s1 < k.seg_end && end < hi) end += tl.segs[s1++].K;
                ok = ok && s1 - s0 <= kTileSegs;
                parts.push_back({s0, s1, lo - pos, hi - pos});
            }
            if (ok || want >= ks[t]) break;
        }
        const int np = (int)parts.size();
        const int64_t nt = (outs[t] + area - 1) / area;
        const int64_t step = std::min<int64_t>(area, 32 * ((outs[t] + 32 * nt - 1) / (32 * nt)));
        for (int64_t o0 = 0; o0 < outs[t]; o0 += step) {
            const int cnt = (int)std::min<int64_t>(step, outs[t] - o0), pad = (cnt + 31) & ~31;
            const int split = np > 1 ? tl.nsplit++ : -1;
            const int64_t base = tl.npartial;
            int64_t row = 0, col = o0;   // of output o0, where a flattened index does not do
            if (outs[t] > kFlatOuts) {
                row = k.herm ? (int64_t)((std::sqrt(8.0 * (double)o0 + 1.0) - 1.0) * 0.5) : o0 / k.N;
                if (k.herm) row += (row + 1) * (row + 2) / 2 <= o0 ? 1 : row * (row + 1) / 2 > o0 ? -1 : 0;
                col = k.herm ? o0 - row * (row + 1) / 2 : o0 - row * k.N;
            }
            if (np > 1) tl.npartial += (int64_t)np * pad;
            for (int p = 0; p < np; ++p) {
                Tile tile{};
                tile.task = (int32_t)t; tile.m0 = (int32_t)row; tile.o0 = (int32_t)col; tile.cnt = cnt; tile.ks = cks;
                tile.N = k.herm ? 0 : k.N;
                tile.seg_lo = parts[p].seg_lo; tile.seg_hi = parts[p].seg_hi;
                tile.k0 = (int32_t)parts[p].k0; tile.k1 = (int32_t)parts[p].k1;
                tile.split = split; tile.part = (uint16_t)p; tile.nparts = (uint16_t)np; tile.split_base = (int32_t)(base / 32);
                tile.cost = (int32_t)std::min<int64_t>((int64_t)cnt * std::max<int64_t>(parts[p].k1 - parts[p].k0, 1), 0x7fffffff);
                tl.tiles.push_back(tile);
            }
        }
    }
    // longest tiles first: the grid drains big work before the tail of small tiles
    std::stable_sort(tl.tiles.begin(), tl.tiles.end(),
                     [](const Tile& a, const Tile& b) { return a.cost > b.cost; });
}

// 16 x 16 tiles of the correction kernel, long K split along segment boundaries into parts of about ksplit
void make_corr_tiles(TaskList& tl, int ksplit) {
    tl.ctiles.clear();
    tl.nsplit = 0;
    tl.npartial = 0;
    constexpr int tm = kTileCorr;
    int parts_total = 0;
    for (size_t t = 0; t < tl.tasks.size(); ++t) {
        const Task& k = tl.tasks[t];
        int64_t ksum = 0;
        for (int s = k.seg_begin; s < k.seg_end; ++s) ksum += tl.segs[s].K;
        std::vector<std::pair<int, int>> parts;
        const int nseg = k.seg_end - k.seg_begin;
        const int want = (int)std::min<int64_t>({(ksum + ksplit - 1) / ksplit, (int64_t)nseg, (int64_t)8});
        if (want <= 1) {
            parts.push_back({k.seg_begin, k.seg_end});
        } else {
            const double target = (double)ksum / want;
            int lo = k.seg_begin;
            int64_t acc = 0;
            for (int s = k.seg_begin; s < k.seg_end; ++s) {
                acc += tl.segs[s].K;
                const bool room = (int)parts.size() < want - 1;
                if (room && acc >= target * (parts.size() + 1) && s + 1 < k.seg_end) {
                    parts.push_back({lo, s + 1});
                    lo = s + 1;
                }
            }
            parts.push_back({lo, k.seg_end});
        }
        for (int m0 = 0; m0 < k.M; m0 += tm)
            for (int n0 = 0; n0 < k.N; n0 += tm) {
                const int mm = std::min(tm, k.M - m0), nn = std::min(tm, k.N - n0);
                const int np = (int)parts.size();
                const int split = np > 1 ? tl.nsplit++ : -1;
                const int base = np > 1 ? parts_total : 0;
                if (np > 1) parts_total += np;
                for (int p = 0; p < np; ++p) {
                    int64_t kp = 0;
                    for (int s = parts[p].first; s < parts[p].second; ++s) kp += tl.segs[s].K;
                    CorrTile tile{};
                    tile.task = (int32_t)t; tile.m0 = m0; tile.n0 = n0;
                    tile.cost = (int32_t)std::min<int64_t>((int64_t)mm * nn * std::max<int64_t>(kp, 1), 0x7fffffff);
                    tile.seg_lo = parts[p].first; tile.seg_hi = parts[p].second;
                    tile.split = split; tile.part = p; tile.nparts = np; tile.split_base = base;
                    tl.ctiles.push_back(tile);
                }
            }
    }
    tl.npartial = (int64_t)parts_total * tm * tm;
    std::stable_sort(tl.ctiles.begin(), tl.ctiles.end(),
                     [](const CorrTile& a, const CorrTile& b) { return a.cost > b.cost; });
}

namespace {

struct PairInfo {
    int qi, ri;
    int64_t off;
    int dl, dr;
};

std::vector<PairInfo> pairs_of(const tdmrg_ctx* c, int a, int b) {
    std::vector<PairInfo> out;
    const Side& L = c->side[0];
    const Side& R = c->side[1];
    int64_t off = 0;
    for (size_t qi = 0; qi < L.dim.size(); ++qi) {
        int ri = R.find(a - L.nup[qi], b - L.ndn[qi]);
        if (ri < 0) continue;
        out.push_back({(int)qi, ri, off, L.dim[qi], R.dim[ri]});
        off += (int64_t)L.dim[qi] * R.dim[ri];
    }
    return out;
}

}  // namespace

int build_plan(tdmrg_ctx* c, const std::vector<Term>& terms, int qa, int qb, int oa, int ob, Plan* p) {
    const Side& L = c->side[0];
    p->qin[0] = qa; p->qin[1] = qb; p->qout[0] = oa; p->qout[1] = ob;
    std::vector<PairInfo> pin = pairs_of(c, qa, qb), pout = pairs_of(c, oa, ob);
    p->n_in = pin.empty() ? 0 : pin.back().off + (int64_t)pin.back().dl * pin.back().dr;
    p->n_out = pout.empty() ? 0 : pout.back().off + (int64_t)pout.back().dl * pout.back().dr;
    std::vector<int> out_of_q(L.dim.size(), -1);
    for (size_t k = 0; k < pout.size(); ++k) out_of_q[pout[k].qi] = (int)k;

    // left sectors that the terms connect: the superblocks of a direct sum stay apart, and every one gets the K parts (so
    // the bits) that it has alone.  Parts by a task's own size would do that too, but are up to 20 % slower (H psi and the
    // ground state at L=16 m=200) where they are not the same.
    std::vector<int> root(L.dim.size());
    for (size_t k = 0; k < root.size(); ++k) root[k] = (int)k;
    auto find_root = [&](int q) {
        while (root[q] != q) q = root[q] = root[root[q]];
        return q;
    };
    std::vector<std::vector<Seg>> direct(pout.size()), left(pout.size());
    std::vector<Task> s1_inter;
    std::vector<Seg> s1_inter_seg;
    std::vector<int> s1_inter_q, g1, g2;   // left sectors of the intermediates, groups of the tasks
    int64_t scr = 0;
    const cplx one = make_double2(1.0, 0.0);

    for (const PairInfo& pi : pin) {
        int nparity = (L.nup[pi.qi] + L.ndn[pi.qi]) & 1;
        for (const Term& t : terms) {
            const BlockOp* A = t.opL >= 0 ? &c->ops[0].at(t.opL) : nullptr;
            const BlockOp* B = t.opR >= 0 ? &c->ops[1].at(t.opR) : nullptr;
            double sgn = (B && B->odd && nparity) ? -1.0 : 1.0;
            // a connection's coefficient is either folded into the segment or read at run time from the
            // caller's device array (tdmrg_set_coefficients); the fermion sign stays static
            const bool run_time = c->dcoef != nullptr && t.conn >= 0;
            cplx sc = run_time ? make_double2(sgn, 0.0) : make_double2(sgn * t.coeff.x, sgn * t.coeff.y);
            const int dcoef = run_time ? t.conn : -1;
            // real operands skip their imaginary products: A (left operator) with a real static factor,
            // B (right operator) always (its factor goes on A in the FP64 kernel)
            const int8_t a_real = (A && A->real && sc.y == 0.0 && dcoef < 0) ? 1 : 0;
            const int8_t b_real = (B && B->real) ? 2 : 0;
            std::vector<std::pair<int, int64_t>> al, bl;
            if (!A) al.push_back({pi.qi, -1});
            else for (auto& blk : A->blocks) if (std::get<1>(blk) == pi.qi) al.push_back({std::get<0>(blk), std::get<2>(blk)});
            if (!B) bl.push_back({pi.ri, -1});
            else for (auto& blk : B->blocks) if (std::get<1>(blk) == pi.ri) bl.push_back({std::get<0>(blk), std::get<2>(blk)});
            for (auto& a : al) {
                int ko = out_of_q[a.first];
                if (ko < 0) continue;
                const PairInfo& po = pout[ko];
                for (auto& b : bl) {
                    if (b.first != po.ri) continue;
                    if (!A && !B) return fail(c, TDMRG_EINVAL, "a term needs an operator on at least one block");
                    root[find_root(a.first)] = find_root(pi.qi);
                    if (!A) {          // Psi'_q += sc * Psi_q B^T, written by stage 1
                        Seg s{};
                        s.a_off = pi.off; s.a_buf = BUF_IN; s.lda = pi.dr;
                        s.b_off = b.second; s.b_buf = BUF_OPS; s.ldb = pi.dr; s.opb = OPB_T;
                        s.K = pi.dr; s.scale = sc; s.dscale = -1; s.dcoef = dcoef;
                        s.rflags = b_real;
                        direct[ko].push_back(s);
                    } else if (!B) {   // Psi'_q += sc * A Psi_{q'}
                        Seg s{};
                        s.a_off = a.second; s.a_buf = BUF_OPS; s.lda = pi.dl;
                        s.b_off = pi.off; s.b_buf = BUF_IN; s.ldb = pi.dr; s.opb = OPB_N;
                        s.K = pi.dl; s.scale = sc; s.dscale = -1; s.dcoef = dcoef;
                        s.rflags = a_real;
                        left[ko].push_back(s);
                    } else {           // T = Psi_{q'} B^T (scratch, stored as T^T), then Psi'_q += sc * A T
                        // T^T rows are the columns of T: the stage-1 stores and the stage-2 operand
                        // reads (slicing of the columns of T) run along contiguous memory
                        Task tk{};
                        tk.c_off = scr; tk.c_buf = BUF_SCRATCH; tk.ldc = pi.dl; tk.M = pi.dl; tk.N = po.dr;
                        tk.beta = 0; tk.trans = 1;
                        Seg s{};
                        s.a_off = pi.off; s.a_buf = BUF_IN; s.lda = pi.dr;
                        s.b_off = b.second; s.b_buf = BUF_OPS; s.ldb = pi.dr; s.opb = OPB_T;
                        s.K = pi.dr; s.scale = one; s.dscale = -1;
                        s.rflags = b_real;
                        s1_inter.push_back(tk);
                        s1_inter_q.push_back(pi.qi);
                        s1_inter_seg.push_back(s);
                        Seg s2{};
                        s2.a_off = a.second; s2.a_buf = BUF_OPS; s2.lda = pi.dl;
                        s2.b_off = scr; s2.b_buf = BUF_SCRATCH; s2.ldb = pi.dl; s2.opb = OPB_T;
                        s2.K = pi.dl; s2.scale = sc; s2.dscale = -1; s2.dcoef = dcoef;
                        s2.rflags = a_real;
                        left[ko].push_back(s2);
                        scr += (int64_t)pi.dl * po.dr;
                    }
                }
            }
        }
    }
    // stage 1: direct writes into the output, then scratch intermediates
    TaskList& s1 = p->stage1;
    TaskList& s2 = p->stage2;
    release(c, s1); release(c, s2);
    s1.tasks.clear(); s1.segs.clear(); s2.tasks.clear(); s2.segs.clear();
    for (size_t k = 0; k < pout.size(); ++k) {
        if (direct[k].empty()) continue;
        Task tk{};
        tk.c_off = pout[k].off; tk.c_buf = BUF_OUT; tk.ldc = pout[k].dr; tk.M = pout[k].dl; tk.N = pout[k].dr;
        tk.beta = 0;
        tk.seg_begin = (int)s1.segs.size();
        for (auto& s : direct[k]) s1.segs.push_back(s);
        tk.seg_end = (int)s1.segs.size();
        s1.tasks.push_back(tk);
        g1.push_back(find_root(pout[k].qi));
    }
    for (size_t k = 0; k < s1_inter.size(); ++k) {
        Task tk = s1_inter[k];
        tk.seg_begin = (int)s1.segs.size();
        s1.segs.push_back(s1_inter_seg[k]);
        tk.seg_end = (int)s1.segs.size();
        s1.tasks.push_back(tk);
        g1.push_back(find_root(s1_inter_q[k]));
    }
    // stage 2: one task per output block that still needs left products or a zero fill
    for (size_t k = 0; k < pout.size(); ++k) {
        bool has_direct = !direct[k].empty();
        if (has_direct && left[k].empty()) continue;
        Task tk{};
        tk.c_off = pout[k].off; tk.c_buf = BUF_OUT; tk.ldc = pout[k].dr; tk.M = pout[k].dl; tk.N = pout[k].dr;
        tk.beta = has_direct ? 1 : 0;
        tk.seg_begin = (int)s2.segs.size();
        for (auto& s : left[k]) s2.segs.push_back(s);
        tk.seg_end = (int)s2.segs.size();
        s2.tasks.push_back(tk);
        g2.push_back(find_root(pout[k].qi));
    }
    p->group[0] = g1;
    p->group[1] = g2;
    make_tiles(s1, &g1);
    make_tiles(s2, &g2);
    p->scratch = scr;
    p->flops = s1.flops + s2.flops;
    int urc = upload(c, s1);
    if (!urc) urc = upload(c, s2);
    if (!urc) urc = uploads_done(c, "plan upload");
    if (urc) return urc;
    if (scr > c->scratch_cap) {
        if (c->scratch) dev_free(c, c->scratch, c->scratch_cap * sizeof(cplx));
        c->scratch = nullptr;
        c->scratch_cap = 0;
        int rc = dev_alloc(c, (void**)&c->scratch, scr * sizeof(cplx), "superblock scratch");
        if (rc) return rc;
        c->scratch_cap = scr;
    }
    return cuda_check(c, cudaGetLastError(), "plan upload");
}

int run_plan(tdmrg_ctx* c, const Plan& p, const cplx* in, cplx* out, const int* skip_flag, int skip_step) {
    if (p.oz.ready) return run_oz(c, p, in, out, skip_flag, skip_step);
    GemmArgs a{};
    a.bufs[BUF_OPS] = c->pool;
    a.bufs[BUF_IN] = const_cast<cplx*>(in);
    a.bufs[BUF_SCRATCH] = c->scratch;
    a.bufs[BUF_OUT] = out;
    a.dscale = c->dscale;
    a.dcoef = c->dcoef;
    for (const TaskList* tl : {&p.stage1, &p.stage2}) {
        if (tl->tiles.empty()) continue;
        a.tasks = tl->d_tasks; a.segs = tl->d_segs; a.tiles = tl->d_tiles; a.ntiles = (int)tl->tiles.size();
        a.partials = tl->d_partials; a.counters = tl->d_counters;
        cudaError_t e = launch_gemm_f64(a, c->stream, skip_flag, skip_step);
        c->launches++;
        int rc = cuda_check(c, e, "superblock product launch");
        if (rc) return rc;
    }
    return TDMRG_OK;
}

}  // namespace tdmrg
