// Grouped complex FP64 GEMM for the sector-pair products of H psi (Sec. IV, Hamiltonian
// connections), the excitation operators (Eq. b), rho_L (Eq. rdensitymatrix) and every other superblock product.
//
// On GB300 FP64 runs at about 1 TFLOP/s for the whole chip (scalar DFMA and the FP64 MMA alike): a warp-wide
// DFMA holds its sub-partition's FP64 pipe for ~64 cycles, an m8n8k4 MMA for ~640, so memory and issue slots
// are nearly free beside the arithmetic, and what decides is how many FP64 instructions are spent and how
// evenly they fall on the 608 pipes.  Hence scalar DFMA with one output per lane:
//   - a tile is a range of a task's outputs in flattened (row-major, for a Hermitian result lower-triangle)
//     order, so blocks of any odd size fill their warps (an 8 x 8 MMA grid leaves 30-60 % of a ragged sector
//     block's MMA work on padding), and K runs over its exact length;
//   - the K range of an output is divided among `ks` groups of warps of the CTA (summed in order through shared
//     memory), and over CTAs when that is not enough, down to a K per warp that keeps every pipe busy
//     (make_tiles): small superblocks are bound by the longest chain of one warp, not by the total;
//   - operands go from global memory (L1 / L2) straight to registers, four k ahead of their use: at 256
//     cycles per complex multiply-add of a warp the loads are hidden without shared memory or barriers;
//   - conjugations and the segment factor are applied once per segment on the accumulated sums.
// Measured: rho_L at L=48 m=1000 564 us (0.60 GFLOP of lower triangles, 1.07 TFLOP/s), H psi at L=8 m=16 8.3 us; as 16 x 16
// tiles of m8n8k4 MMAs, each warp one 8 x 8 block over the whole K, 872 and 17.7 us.
// CTAs that share a K split store partial sums; the last part to arrive (atomic ticket) sums all parts in index
// order, so results do not depend on scheduling.
//
// The correction kernel serves the update W' = (I + D) W of the eigen-refinement, where D is small
// (|D| <= 1e-3, ~1e-7 in the last iteration): D W runs in FP32 (each CTA accumulates one K part of at
// most a few dozen terms; parts are summed in FP64), so its rounding is ~1e-7 of |D| |W|, and the
// epilogue adds W itself in FP64.  W is the B operand of the task's first segment.  FP32 accumulation
// is what limits the accuracy, so it suits small corrections only, not full products.  It works on 16 x 16
// output tiles staged through shared memory.
#include "internal.h"
#include "lane_mac.cuh"

namespace tdmrg {
namespace {

constexpr int GT = 256;               // threads of a CTA of the grouped GEMM

// Sign flip of a double on the integer pipe
__device__ __forceinline__ double neg(double x) { return __longlong_as_double(__double_as_longlong(x) ^ (1ll << 63)); }

// One segment as the lanes read it: A(m, k) at a[m * am + k * ak], B(k, n) at b[n * bn + k * bk].
struct SegView {
    const double2* a;
    const double2* b;
    int am, ak, bn, bk;
    int K, mode;                      // mode 0 complex, 1 A real, 2 B real
    double ca, cb;                    // -1: conjugated operand
    double sr, si;                    // factor
};

__global__ void __launch_bounds__(GT, 2) gemm_f64_kernel(GemmArgs args, const int* skip_flag, int skip_step) {
    __shared__ SegView sv[kTileSegs];
    __shared__ double2 red[GT];
    __shared__ int last;
    // the tables before the wait for the previous kernel: they are the plan's, no kernel writes them
    const Tile tile = args.tiles[blockIdx.x];
    const Task task = args.tasks[tile.task];   // used at the end only
    const int tid = threadIdx.x;
    const int nseg = tile.seg_hi - tile.seg_lo;
    Seg seg{};
    if (tid < nseg) seg = args.segs[tile.seg_lo + tid];
    pdl_enter();
    if (skip_flag != nullptr && skip_step >= *skip_flag) return;   // Krylov space already complete
    if (tid < nseg) {
        SegView w;
        w.a = args.bufs[seg.a_buf] + seg.a_off;
        w.b = args.bufs[seg.b_buf] + seg.b_off;
        w.am = seg.opa ? 1 : seg.lda; w.ak = seg.opa ? seg.lda : 1;
        const bool nb = seg.opb == OPB_N || seg.opb == OPB_CN;
        w.bn = nb ? 1 : seg.ldb; w.bk = nb ? seg.ldb : 1;
        w.K = seg.K;
        w.mode = (seg.rflags & 1) ? 1 : (seg.rflags & 2) ? 2 : 0;
        w.ca = seg.opa == 2 ? -1.0 : 1.0;
        w.cb = (seg.opb == OPB_C || seg.opb == OPB_CN) ? -1.0 : 1.0;
        double sr = seg.scale.x, si = seg.scale.y;
        if (seg.dscale >= 0) {
            const double d = args.dscale[seg.dscale];
            sr *= d; si *= d;
        }
        if (seg.dcoef >= 0 && args.dcoef != nullptr) {   // run-time coefficient of a connection term
            const cplx d = args.dcoef[seg.dcoef];
            const double tr = sr * d.x - si * d.y;
            si = sr * d.y + si * d.x;
            sr = tr;
        }
        w.sr = sr; w.si = si;
        sv[tid] = w;
    }
    // this thread's output and its share of the K range (uniform per warp)
    const int pad = (tile.cnt + 31) & ~31;
    const int part = tid / pad, lo = tid - part * pad;
    const bool active = part < tile.ks && lo < tile.cnt;
    int m = 0, n = 0;
    if (active) {
        const int o = tile.o0 + lo;
        if (tile.N != 0) {
            m = o / tile.N;
            n = o - m * tile.N;
            m += tile.m0;
        } else if (tile.m0 == 0) {   // row m of the lower triangle starts at m (m + 1) / 2
            m = (int)((sqrtf(8.f * (float)o + 1.f) - 1.f) * 0.5f);
            while ((m + 1) * (m + 2) / 2 <= o) ++m;
            while (m * (m + 1) / 2 > o) --m;
            n = o - m * (m + 1) / 2;
        } else {
            m = tile.m0;
            n = o;
            while (n > m) n -= ++m;
        }
    }
    const int kspan = tile.k1 - tile.k0;
    const int ka = tile.k0 + kspan * part / tile.ks, kb = tile.k0 + kspan * (part + 1) / tile.ks;
    __syncthreads();
    double re = 0.0, im = 0.0;
    if (active) {
        int pos = 0;   // k of the tile's first segment's start; tile.k0 and k1 count from there
        for (int s = 0; s < nseg && pos < kb; ++s) {
            const SegView& w = sv[s];
            const int k0 = max(ka - pos, 0), k1 = min(kb - pos, w.K);
            pos += w.K;
            if (k0 >= k1) continue;
            const double2* pa = w.a + (int64_t)m * w.am + (int64_t)k0 * w.ak;
            const double2* pb = w.b + (int64_t)n * w.bn + (int64_t)k0 * w.bk;
            double q[4] = {0.0, 0.0, 0.0, 0.0};
            if (w.mode == 0) seg_mac<0, 4>(pa, pb, w.ak, w.bk, k1 - k0, q);
            else if (w.mode == 1) seg_mac<1, 4>(pa, pb, w.ak, w.bk, k1 - k0, q);
            else seg_mac<2, 4>(pa, pb, w.ak, w.bk, k1 - k0, q);
            const double pr = fma(-w.ca * w.cb, q[1], q[0]), pi = fma(w.cb, q[2], w.ca * q[3]);
            const double sr = w.sr, si = w.si;
            if (si == 0.0) {
                re = fma(sr, pr, re);
                im = fma(sr, pi, im);
            } else {
                re = fma(sr, pr, fma(-si, pi, re));
                im = fma(sr, pi, fma(si, pr, im));
            }
        }
    }
    if (tile.ks > 1) {   // the K shares of this CTA, summed in order
        if (active && part > 0) red[tid] = make_double2(re, im);
        __syncthreads();
        if (active && part == 0)
            for (int p = 1; p < tile.ks; ++p) {
                const double2 x = red[p * pad + lo];
                re += x.x; im += x.y;
            }
    }
    const bool out = active && part == 0;
    if (tile.split >= 0) {
        // split-K over CTAs: publish this part, the last part to arrive sums all parts in index order
        cplx* base = args.partials + 32 * (int64_t)tile.split_base;
        if (out) base[(int64_t)tile.part * pad + lo] = make_double2(re, im);
        __threadfence();
        __syncthreads();
        if (tid == 0) last = (atomicAdd(args.counters + tile.split, 1) == tile.nparts - 1);
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (out) {
            re = 0.0; im = 0.0;
            for (int p = 0; p < tile.nparts; ++p) {
                const double2 x = __ldcg(base + (int64_t)p * pad + lo);
                re += x.x; im += x.y;
            }
        }
        if (tid == 0) args.counters[tile.split] = 0;   // ready for the next launch
    }
    if (!out) return;
    cplx* __restrict__ C = args.bufs[task.c_buf] + task.c_off;
    cplx* p = task.trans ? C + (int64_t)n * task.ldc + m : C + (int64_t)m * task.ldc + n;
    if (task.beta) {
        const double2 o = *p;
        re += o.x;
        im += o.y;
    }
    *p = make_double2(re, im);
    if (task.herm && m != n) C[(int64_t)n * task.ldc + m] = make_double2(re, neg(im));
}

// ---- correction kernel: C = (I + D) W on 16 x 16 tiles --------------------------------------------
constexpr int TS = kTileCorr;    // 16
constexpr int KC = 16;
constexpr int PAD = TS + 4;      // row stride of the staged planes (conflict-free fragment loads)

// acc += a * b for complex a = (ar, ai), b = (br, bi) in FP32
__device__ __forceinline__ void cfma32(float& cr, float& ci, float ar, float ai, float br, float bi) {
    cr = fmaf(ar, br, fmaf(-ai, bi, cr));
    ci = fmaf(ar, bi, fmaf(ai, br, ci));
}

__global__ void __launch_bounds__(128) gemm_corr_kernel(GemmArgs args, const int* skip_flag, int skip_step) {
    pdl_enter();
    if (skip_flag != nullptr && skip_step >= *skip_flag) return;
    __shared__ float fA[2][TS][PAD], fB[2][KC][PAD];   // [0] real and [1] imaginary
    __shared__ int last;
    const CorrTile tile = args.ctiles[blockIdx.x];
    const Task task = args.tasks[tile.task];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int gid = lane >> 2, tig = lane & 3;
    const int m0 = tile.m0, n0 = tile.n0;
    const int Mt = min(TS, task.M - m0), Nt = min(TS, task.N - n0);
    // warp w owns the 8 x 8 sub-block (w / 2, w % 2)
    const int bi = warp >> 1, bj = warp & 1;
    const bool active = (8 * bi < Mt) && (8 * bj < Nt);
    float fre[2] = {0.f, 0.f}, fim[2] = {0.f, 0.f};
    for (int s = tile.seg_lo; s < tile.seg_hi; ++s) {
        const Seg seg = args.segs[s];
        const cplx* __restrict__ A = args.bufs[seg.a_buf] + seg.a_off;
        const cplx* __restrict__ B = args.bufs[seg.b_buf] + seg.b_off;
        for (int k0 = 0; k0 < seg.K; k0 += KC) {
            const int kc = min(KC, seg.K - k0);
#pragma unroll
            for (int u = 0; u < 2; ++u) {             // A chunk TS x KC: threads along k
                const int e = tid + 128 * u, r = e / KC, k = e % KC;
                double2 v = make_double2(0.0, 0.0);
                if (r < Mt && k < kc) v = A[(int64_t)(m0 + r) * seg.lda + k0 + k];
                fA[0][r][k] = (float)v.x;
                fA[1][r][k] = (float)v.y;
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {             // B[k][n] at B[k*ldb + n]: threads along n
                const int e = tid + 128 * u, k = e / TS, n = e % TS;
                double2 v = make_double2(0.0, 0.0);
                if (k < kc && n < Nt) v = B[(int64_t)(k0 + k) * seg.ldb + n0 + n];
                fB[0][k][n] = (float)v.x;
                fB[1][k][n] = (float)v.y;
            }
            __syncthreads();
            if (active) {
                const int rr = 8 * bi + gid;
                for (int kk = 0; kk < kc; ++kk) {
                    const float ar = fA[0][rr][kk], ai = fA[1][rr][kk];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int cc = 8 * bj + 2 * tig + e;
                        cfma32(fre[e], fim[e], ar, ai, fB[0][kk][cc], fB[1][kk][cc]);
                    }
                }
            }
            __syncthreads();
        }
    }
    // this thread's two outputs: row 8 bi + gid, columns 8 bj + 2 tig + e
    const int r = 8 * bi + gid, col0 = 8 * bj + 2 * tig;
    double2 v[2] = {make_double2((double)fre[0], (double)fim[0]), make_double2((double)fre[1], (double)fim[1])};
    if (tile.split >= 0) {
        cplx* part = args.partials + ((int64_t)tile.split_base + tile.part) * (TS * TS);
        if (active) {
            part[r * TS + col0] = v[0];
            part[r * TS + col0 + 1] = v[1];
        }
        __threadfence();
        __syncthreads();
        if (tid == 0) last = (atomicAdd(args.counters + tile.split, 1) == tile.nparts - 1);
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (active) {
            const cplx* base = args.partials + (int64_t)tile.split_base * (TS * TS);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                double2 t = make_double2(0.0, 0.0);
                for (int p = 0; p < tile.nparts; ++p) {
                    const double2 x = __ldcg(base + (int64_t)p * (TS * TS) + r * TS + col0 + e);
                    t.x += x.x; t.y += x.y;
                }
                v[e] = t;
            }
        }
        if (tid == 0) args.counters[tile.split] = 0;   // ready for the next launch
    }
    if (!active) return;
    cplx* __restrict__ C = args.bufs[task.c_buf] + task.c_off;
    const Seg s0 = args.segs[task.seg_begin];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int col = col0 + e;
        if (r < Mt && col < Nt) {   // (I + D) W: add W in FP64
            const double2 w = args.bufs[s0.b_buf][s0.b_off + (int64_t)(m0 + r) * s0.ldb + n0 + col];
            C[(int64_t)(m0 + r) * task.ldc + n0 + col] = make_double2(v[e].x + w.x, v[e].y + w.y);
        }
    }
}

}  // namespace

cudaError_t launch_gemm_f64(const GemmArgs& a, cudaStream_t s, const int* skip_flag, int skip_step) {
    if (a.ntiles <= 0) return cudaSuccess;
    launch_pdl(gemm_f64_kernel, a.ntiles, GT, 0, s, a, skip_flag, skip_step);
    return cudaGetLastError();
}

cudaError_t launch_gemm_corr(const GemmArgs& a, cudaStream_t s, const int* skip_flag, int skip_step) {
    if (a.ntiles <= 0) return cudaSuccess;
    launch_pdl(gemm_corr_kernel, a.ntiles, 128, 0, s, a, skip_flag, skip_step);
    return cudaGetLastError();
}

}  // namespace tdmrg
