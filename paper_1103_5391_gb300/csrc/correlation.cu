// Correlation grid <phi1| A_i B_j |phi2> over a list of left operators A_i and right operators B_j: the
// two-state form of Eq. generalcorrelation with one local operator per block, e.g. the Green's function
// G_ij(t) = <phi(t)| c_i c^dag_j |psi(t)> (Sec. I) measured on device-resident states.
//
// The grid factorises: with T_j = s phi2 B_j^T (s the fermion sign) and Z_i = A_i^dag phi1, both on the blocks (q', r) of
// left input sectors q' and right output sectors r,
//     <phi1| A_i B_j |phi2> = sum over blocks of <Z_i(q', r), T_j(q', r)>,
// so nL + nR products, one grouped FP64 launch (they do not depend on one another), and nL nR dots replace the 2 nL nR
// products of the entries taken one by one: at L=32 m=400 with a 4 x 4 grid 134 instead of 482 us.  Every Z_i and T_j is a
// vector over the same block list (absent blocks stay zero), so an entry is one plain dot: partials over kCorrChunks
// chunks, summed in chunk order.
#include <algorithm>
#include <vector>

#include "internal.h"

namespace tdmrg {
namespace {

constexpr int CT = 256;

// part[p * kCorrChunks + chunk] = sum over the chunk of conj(Z_i) T_j, p = i nR + j
__global__ void __launch_bounds__(CT) k_corr_dots(const cplx* __restrict__ Z, const cplx* __restrict__ T, int nR, int64_t n,
                                                  double2* __restrict__ part) {
    pdl_enter();
    const int p = blockIdx.x, ch = blockIdx.y;
    const int64_t len = (n + kCorrChunks - 1) / kCorrChunks;
    const int64_t lo = min(n, (int64_t)ch * len), hi = min(n, lo + len);
    const cplx* __restrict__ z = Z + (int64_t)(p / nR) * n;
    const cplx* __restrict__ w = T + (int64_t)(p % nR) * n;
    double sr = 0.0, si = 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += CT) {
        const double2 a = z[i], b = w[i];
        sr = fma(a.x, b.x, fma(a.y, b.y, sr));
        si = fma(a.x, b.y, fma(-a.y, b.x, si));
    }
    __shared__ double2 sh[CT / 32];
    for (int o = 16; o > 0; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = make_double2(sr, si);
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 t = make_double2(0.0, 0.0);
        for (int k = 0; k < CT / 32; ++k) { t.x += sh[k].x; t.y += sh[k].y; }
        part[(int64_t)p * kCorrChunks + ch] = t;
    }
}

// blocks of a state copied into a Z_i or T_j whose operator is the identity (CorrCopy: element offsets and length)
__global__ void __launch_bounds__(CT) k_corr_copy(const CorrCopy* __restrict__ copies, const cplx* __restrict__ phi1,
                                                  const cplx* __restrict__ phi2, cplx* __restrict__ Z, cplx* __restrict__ T) {
    pdl_enter();
    const CorrCopy c = copies[blockIdx.x];
    const cplx* __restrict__ src = (c.right ? phi2 : phi1) + c.src;
    cplx* __restrict__ dst = (c.right ? T : Z) + c.dst;
    for (int64_t i = threadIdx.x; i < c.len; i += CT) dst[i] = src[i];
}

__global__ void k_corr_final(const double2* __restrict__ part, int npairs, cplx* __restrict__ out) {
    pdl_enter();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npairs) return;
    double2 t = make_double2(0.0, 0.0);
    for (int k = 0; k < kCorrChunks; ++k) { t.x += part[(int64_t)p * kCorrChunks + k].x; t.y += part[(int64_t)p * kCorrChunks + k].y; }
    out[p] = t;
}

void free_corr(tdmrg_ctx* c, CorrPlan& cp) {
    release(c, cp.tl);
    dev_free(c, cp.Z, (size_t)cp.nL * cp.n * sizeof(cplx));
    dev_free(c, cp.T, (size_t)cp.nR * cp.n * sizeof(cplx));
    dev_free(c, cp.part, (size_t)cp.nL * cp.nR * kCorrChunks * sizeof(double2));
    dev_free(c, cp.copies, (size_t)cp.ncopies * sizeof(CorrCopy));
}

// Blocks (q', r) of the grid: every left input sector q' (with a partner in Q2) and right output sector r (with a
// partner in Q1) that some A_i and some B_j connect; the products of Z_i and T_j on them.
int build_corr(tdmrg_ctx* c, int nL, const int32_t* opL, int nR, const int32_t* opR, int a1, int b1, int a2, int b2, CorrPlan& cp) {
    const Side& L = c->side[0];
    const Side& R = c->side[1];
    const int sl = (int)L.dim.size(), sr = (int)R.dim.size();
    std::vector<int64_t> off1(sl, -1), off2(sl, -1);   // offsets of the blocks of left sector q in phi1 and phi2
    std::vector<int> r1(sl, -1), r2(sl, -1), q1(sr, -1);
    int64_t o1 = 0, o2 = 0;
    for (int q = 0; q < sl; ++q) {
        r1[q] = R.find(a1 - L.nup[q], b1 - L.ndn[q]);
        r2[q] = R.find(a2 - L.nup[q], b2 - L.ndn[q]);
        if (r1[q] >= 0) { off1[q] = o1; o1 += (int64_t)L.dim[q] * R.dim[r1[q]]; q1[r1[q]] = q; }
        if (r2[q] >= 0) { off2[q] = o2; o2 += (int64_t)L.dim[q] * R.dim[r2[q]]; }
    }
    // (q', r) -> operator block offset (-1: identity), per operator
    typedef std::map<std::pair<int, int>, int64_t> Blocks;
    std::vector<Blocks> zb(nL), tb(nR);
    for (int i = 0; i < nL; ++i) {   // A_i[q <- q'] reaches r, the partner of q in Q1
        if (opL[i] < 0) {
            for (int q = 0; q < sl; ++q) if (r1[q] >= 0) zb[i][{q, r1[q]}] = -1;
        } else {
            for (const auto& blk : c->ops[0].at(opL[i]).blocks)
                if (r1[std::get<0>(blk)] >= 0) zb[i][{std::get<1>(blk), r1[std::get<0>(blk)]}] = std::get<2>(blk);
        }
    }
    for (int j = 0; j < nR; ++j) {   // B_j[r <- r'] starts from r', the partner of q' in Q2
        for (int q = 0; q < sl; ++q) {
            if (r2[q] < 0) continue;
            if (opR[j] < 0) {
                tb[j][{q, r2[q]}] = -1;
            } else {
                for (const auto& blk : c->ops[1].at(opR[j]).blocks)
                    if (std::get<1>(blk) == r2[q]) tb[j][{q, std::get<0>(blk)}] = std::get<2>(blk);
            }
        }
    }
    Blocks common;   // -> offset in the Z_i and T_j
    for (const Blocks& t : tb)
        for (const auto& kv : t)
            for (const Blocks& z : zb)
                if (z.count(kv.first)) { common[kv.first] = 0; break; }
    cp.n = 0;
    for (auto& kv : common) {
        kv.second = cp.n;
        cp.n += (int64_t)L.dim[kv.first.first] * R.dim[kv.first.second];
    }
    cp.nL = nL;
    cp.nR = nR;
    std::vector<CorrCopy> copies;
    const cplx one = make_double2(1.0, 0.0);
    auto add = [&](int buf, int64_t dst, int M, int N, const Seg& sg) {
        Task t{};
        t.c_off = dst; t.c_buf = (int8_t)buf; t.ldc = N; t.M = M; t.N = N; t.beta = 0;
        t.seg_begin = (int)cp.tl.segs.size();
        cp.tl.segs.push_back(sg);
        t.seg_end = t.seg_begin + 1;
        cp.tl.tasks.push_back(t);
    };
    for (int i = 0; i < nL; ++i)
        for (const auto& kv : zb[i]) {
            const auto at = common.find(kv.first);
            if (at == common.end()) continue;
            const int qp = kv.first.first, r = kv.first.second, q = q1[r];
            const int64_t dst = (int64_t)i * cp.n + at->second;
            if (kv.second < 0) {
                copies.push_back({off1[q], dst, (int64_t)L.dim[q] * R.dim[r], 0});
                continue;
            }
            Seg sg{};   // A^dag Psi1_q
            sg.a_off = kv.second; sg.a_buf = BUF_OPS; sg.lda = L.dim[qp]; sg.opa = 2;
            sg.b_off = off1[q]; sg.b_buf = BUF_EXTRA0; sg.ldb = R.dim[r]; sg.opb = OPB_N;
            sg.K = L.dim[q]; sg.scale = one; sg.dscale = -1;
            sg.rflags = c->ops[0].at(opL[i]).real ? 1 : 0;
            add(BUF_OUT, dst, L.dim[qp], R.dim[r], sg);
        }
    for (int j = 0; j < nR; ++j)
        for (const auto& kv : tb[j]) {
            const auto at = common.find(kv.first);
            if (at == common.end()) continue;
            const int qp = kv.first.first, r = kv.first.second, rp = r2[qp];
            const int64_t dst = (int64_t)j * cp.n + at->second;
            if (kv.second < 0) {
                copies.push_back({off2[qp], dst, (int64_t)L.dim[qp] * R.dim[rp], 1});
                continue;
            }
            const BlockOp& B = c->ops[1].at(opR[j]);
            Seg sg{};   // (+-) Psi2_{q'} B^T
            sg.a_off = off2[qp]; sg.a_buf = BUF_IN; sg.lda = R.dim[rp];
            sg.b_off = kv.second; sg.b_buf = BUF_OPS; sg.ldb = R.dim[rp]; sg.opb = OPB_T;
            sg.K = R.dim[rp]; sg.dscale = -1;
            sg.scale = make_double2(B.odd && ((L.nup[qp] + L.ndn[qp]) & 1) ? -1.0 : 1.0, 0.0);
            sg.rflags = B.real ? 2 : 0;
            add(BUF_SCRATCH, dst, L.dim[qp], R.dim[r], sg);
        }
    make_tiles(cp.tl);
    int rc = upload(c, cp.tl);
    if (!rc) rc = dev_alloc(c, (void**)&cp.Z, (size_t)nL * cp.n * sizeof(cplx), "correlation vectors");
    if (!rc) rc = dev_alloc(c, (void**)&cp.T, (size_t)nR * cp.n * sizeof(cplx), "correlation vectors");
    if (!rc) rc = dev_alloc(c, (void**)&cp.part, (size_t)nL * nR * kCorrChunks * sizeof(double2), "correlation partials");
    // blocks that an operator does not have stay zero
    if (!rc && cp.Z) rc = cuda_check(c, cudaMemsetAsync(cp.Z, 0, (size_t)nL * cp.n * sizeof(cplx), c->stream), "correlation vectors");
    if (!rc && cp.T) rc = cuda_check(c, cudaMemsetAsync(cp.T, 0, (size_t)nR * cp.n * sizeof(cplx), c->stream), "correlation vectors");
    if (!rc && !copies.empty()) {
        cp.ncopies = (int)copies.size();
        rc = dev_alloc(c, (void**)&cp.copies, copies.size() * sizeof(CorrCopy), "correlation copies");
        if (!rc) rc = cuda_check(c, cudaMemcpy(cp.copies, copies.data(), copies.size() * sizeof(CorrCopy), cudaMemcpyHostToDevice),
                                 "correlation copies");
    }
    if (!rc) rc = uploads_done(c, "correlation upload");
    return rc;
}

}  // namespace

void release_corr(tdmrg_ctx* c) {
    for (auto& kv : c->corr_plans) free_corr(c, *kv.second);
    c->corr_plans.clear();
}

}  // namespace tdmrg

using namespace tdmrg;

extern "C" int tdmrg_correlation(tdmrg_ctx* c, int nL, const int32_t* opL, int nR, const int32_t* opR, int a1, int b1,
                                 const tdmrg_c64* phi1, int a2, int b2, const tdmrg_c64* phi2, tdmrg_c64* out) {
    if (!c) return fail(nullptr, TDMRG_EINVAL, "null context");
    if (nL < 1 || nR < 1 || !opL || !opR || !phi1 || !phi2 || !out) return fail(c, TDMRG_EINVAL, "correlation: bad argument");
    if (!c->side[0].set || !c->side[1].set) return fail(c, TDMRG_ESTATE, "correlation: blocks not set");
    for (int i = 0; i < nL; ++i)
        if (opL[i] >= 0 && !c->ops[0].count(opL[i])) return fail(c, TDMRG_EINVAL, "correlation: left op id not set");
    for (int j = 0; j < nR; ++j)
        if (opR[j] >= 0 && !c->ops[1].count(opR[j])) return fail(c, TDMRG_EINVAL, "correlation: right op id not set");
    for (int i = 0; i < nL; ++i)
        for (int j = 0; j < nR; ++j)
            if (opL[i] < 0 && opR[j] < 0) return fail(c, TDMRG_EINVAL, "correlation: a product with two identities");
    const int64_t n1 = sector_size(c, a1, b1);
    if (n1 == 0 || sector_size(c, a2, b2) == 0) return fail(c, TDMRG_ESECTOR, "correlation: empty sector");
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != c->opts.device) cudaSetDevice(c->opts.device);
    std::vector<int> key{nL, nR, a1, b1, a2, b2};
    key.insert(key.end(), opL, opL + nL);
    key.insert(key.end(), opR, opR + nR);
    auto it = c->corr_plans.find(key);
    int rc = TDMRG_OK;
    if (it == c->corr_plans.end()) {
        std::unique_ptr<CorrPlan> cp(new CorrPlan());
        rc = build_corr(c, nL, opL, nR, opR, a1, b1, a2, b2, *cp);
        if (rc) {
            free_corr(c, *cp);
            if (prev >= 0 && prev != c->opts.device) cudaSetDevice(prev);
            return rc;
        }
        it = c->corr_plans.emplace(key, std::move(cp)).first;
    }
    CorrPlan& cp = *it->second;
    GemmArgs g{};
    g.bufs[BUF_OPS] = c->pool;
    g.bufs[BUF_IN] = (cplx*)phi2;
    g.bufs[BUF_EXTRA0] = (cplx*)phi1;
    g.bufs[BUF_SCRATCH] = cp.T;
    g.bufs[BUF_OUT] = cp.Z;
    g.dscale = c->dscale;
    if (!cp.tl.tiles.empty()) {
        g.tasks = cp.tl.d_tasks; g.segs = cp.tl.d_segs; g.tiles = cp.tl.d_tiles; g.ntiles = (int)cp.tl.tiles.size();
        g.partials = cp.tl.d_partials; g.counters = cp.tl.d_counters;
        c->launches++;
        rc = cuda_check(c, launch_gemm_f64(g, c->stream, nullptr, 0), "correlation products");
    }
    if (!rc && cp.ncopies) {
        launch_pdl(k_corr_copy, cp.ncopies, CT, 0, c->stream, (const CorrCopy*)cp.copies, (const cplx*)phi1, (const cplx*)phi2, cp.Z, cp.T);
        c->launches++;
    }
    if (!rc) {
        const int npairs = nL * nR;
        launch_pdl(k_corr_dots, dim3(npairs, kCorrChunks), CT, 0, c->stream, (const cplx*)cp.Z, (const cplx*)cp.T, nR, cp.n, cp.part);
        launch_pdl(k_corr_final, (npairs + 127) / 128, 128, 0, c->stream, (const double2*)cp.part, npairs, (cplx*)out);
        c->launches += 2;
        rc = cuda_check(c, cudaGetLastError(), "correlation dots");
    }
    if (prev >= 0 && prev != c->opts.device) cudaSetDevice(prev);
    return rc;
}
