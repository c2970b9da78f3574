// Krylov time evolution on the device (Sec. II.A, Eq. lanczosevolution; Sec. II.C,
// Eq. lanczosevolution2; time targets of Sec. II.B).
//
// Lanczos is started from phi itself: v_0 = phi / ||phi||.  Step j: w = H v_j (grouped superblock
// product), then two classical Gram-Schmidt passes: the first removes the alpha_j v_j and beta_j v_{j-1} components (H v_j
// has none above rounding along the others), its dots in FP32; the second, in FP64 against v_0..v_j, removes what it
// leaves, a third the rest where that is most of the vector; alpha_j is the sum of the passes' coefficients,
// beta_{j+1} = ||w||, v_{j+1} = w / beta_{j+1}.  All in one cooperative launch per step, whose blocks exchange partial
// sums twice; the recursion stops at n_K vectors or when beta_{j+1} <= tol * max(1, |alpha_j|).  Then the
// coefficients c_x = ||phi|| e^{-i T t_x} e_0 (= ||phi|| [S^dag e^{-i D t_x} S]_{.,0} with T = S^dag D S)
// are computed on the tridiagonal itself (Taylor series on short substeps, FP64; for equally spaced
// times by powers of the step exponential) and the targets phi(t_x) = sum_k v_k c_x[k] are formed in
// one pass over V.  The vectors, alpha and beta are FP64-accurate and stay on the device; reductions use
// a fixed grid and a fixed summation order, so results do not depend on scheduling.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.h"

namespace tdmrg {
namespace {

constexpr int NB = kRedBlocks;   // reduction blocks
constexpr int kCoefWords = (16 + 32) * 32;   // Krylov coefficients of 16 targets + step exponential columns
constexpr int kBarWords = 4;                  // exponential ticket in word 2
constexpr int NT = 256;          // threads per reduction block
enum { T_ALPHA = 0, T_BETA = 32, T_BETA0 = 64, T_RESID = 65, T_ERR = 66, T_EMIN = 67 };

__device__ __forceinline__ void chunk_of(int64_t n, int64_t& lo, int64_t& hi) {
    const int64_t ch = (n + NB - 1) / NB;
    lo = min(n, (int64_t)blockIdx.x * ch);
    hi = min(n, lo + ch);
}

// Deterministic block sum of a double2 (fixed butterfly, fixed warp order).
__device__ double2 block_sum(double2 v) {
    __shared__ double2 sh[NT / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double2 s = make_double2(0.0, 0.0);
    for (int k = 0; k < NT / 32; ++k) { s.x += sh[k].x; s.y += sh[k].y; }
    return s;   // every thread holds the block total
}

// Sum of part[0..NB-1] by one warp in a fixed order (identical in every block that calls it).
__device__ double2 warp_total(const double2* __restrict__ part) {
    const int l = threadIdx.x & 31;
    double2 s = make_double2(0.0, 0.0);
    for (int b = l; b < NB; b += 32) { s.x += part[b].x; s.y += part[b].y; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
    return s;
}

// h[k] = sum of partials of vector k, for k < nv; every block computes the same values.
__device__ void reduce_coeffs(const double2* __restrict__ part, int nv, double2* h) {
    const int w = threadIdx.x >> 5;
    for (int k = w; k < nv; k += NT / 32) {
        double2 s = warp_total(part + (int64_t)k * NB);
        if ((threadIdx.x & 31) == 0) h[k] = s;
    }
    __syncthreads();
}

__device__ __forceinline__ double2 cdotc(double2 a, double2 b) {   // conj(a) * b
    return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

__global__ void __launch_bounds__(NT) k_norm2(const cplx* __restrict__ x, int64_t n, double2* __restrict__ part) {
    pdl_enter();
    int64_t lo, hi;
    chunk_of(n, lo, hi);
    double s = 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += NT) { const double2 v = x[i]; s += v.x * v.x + v.y * v.y; }
    double2 t = block_sum(make_double2(s, 0.0));
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

// The partial-sum slots of the orthogonalisation steps, emptied before a Lanczos run (rows of grid blocks: the first
// pass's two, then both buffers of the second and of the third pass's).
struct OrthSlots { double2 *partA, *partB[2], *partC[2]; int rows, grid; };
__device__ __forceinline__ void clear_slots(const OrthSlots& sl) {
    const double e = __longlong_as_double(0x7ff4dead7ff4deadll);
    const int n = sl.rows * sl.grid;
    for (int i = blockIdx.x * NT + threadIdx.x; i < n; i += gridDim.x * NT) {
        sl.partB[0][i] = make_double2(e, e);
        sl.partB[1][i] = make_double2(e, e);
        sl.partC[0][i] = make_double2(e, e);
        sl.partC[1][i] = make_double2(e, e);
        if (i < 2 * sl.grid) sl.partA[i] = make_double2(e, e);
    }
}

__global__ void __launch_bounds__(NT) k_init_v0(const cplx* __restrict__ phi, int64_t n, const double2* __restrict__ part,
                                                 cplx* __restrict__ v0, double* __restrict__ tri, int* __restrict__ flags,
                                                 int nk, OrthSlots slots) {
    pdl_enter();
    clear_slots(slots);
    __shared__ double sb[2];
    if (threadIdx.x < 32) {   // one square root and one division per block: each is ~20 FP64 instructions of 64 cycles
        const double2 t = warp_total(part);
        if (threadIdx.x == 0) {
            sb[0] = sqrt(t.x);
            sb[1] = sb[0] > 0.0 ? 1.0 / sb[0] : 0.0;
        }
    }
    __syncthreads();
    const double b0 = sb[0], inv = sb[1];
    int64_t lo, hi;
    chunk_of(n, lo, hi);
    for (int64_t i = lo + threadIdx.x; i < hi; i += NT) { const double2 v = phi[i]; v0[i] = make_double2(v.x * inv, v.y * inv); }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        tri[T_BETA0] = b0;
        tri[T_RESID] = 0.0;
        flags[0] = b0 > 0.0 ? nk : 0;
    }
}

// ---- one Lanczos orthogonalisation step in a single cooperative launch -----------------------
// Two exchanges of partial sums between all blocks separate: (A) the first-pass dots h1_k = <v_k|w>; (B) w' = w -
// sum h1_k v_k, the second-pass dots h2_k = <v_k|w'> and ||w'||^2; (C) beta = ||w' - sum h2_k v_k|| and
// v_{j+1} = (w' - sum h2_k v_k) / beta.  Since h2 holds the projections of w' on orthonormal v_k,
// ||w' - sum h2_k v_k||^2 = ||w'||^2 - sum |h2_k|^2 (h2 is at the FP32 rounding level of the first pass, so
// the difference loses nothing), which saves the exchange of a separate norm pass.  Every block
// reduces the partials of all blocks in the same fixed order, so results do not depend on scheduling.
// Where h2 is more than half of w' all the same (|alpha| above ~1e7 beta: a large constant in H), one pass in FP64 is
// not enough, as the orthogonality lost would grow by |h2| / beta at every step: (B) and (C) are then done once more on
// w' - sum h2_k v_k, with slots of their own.  Without that a spectrum of width 1e-8 around 1 gave Lanczos vectors without
// any orthogonality after five steps.
//
// What bounds it is FP64 issue (a warp-wide FP64 instruction holds a sub-partition ~64 cycles) and, for short vectors,
// the chain of latencies.  Hence:
//   - the block's slices of w and of the newest Krylov vectors come into shared memory by bulk copies issued at the
//     start and are read from there by all three passes (what does not fit is read from global memory);
//   - blocks own whole multiples of 128 elements (four warps' worth, one per sub-partition), no more blocks than that
//     gives: fewer partials for every block to sum;
//   - the second-pass dots are split over the warps by vector, not by element: a warp's five FP64 shuffle-adds then serve
//     all of the block's elements, and no cross-warp sum follows;
//   - a partial sum is its own flag: its slot holds a NaN pattern that no arithmetic produces until the block stores the
//     value, and readers poll the values themselves.  Against a counter barrier this saves the arrival's round trip
//     twice.  Slots are cleared a phase later, when every block is known to have read them.
// Polls are bounded: when one runs out the kernel sets a status bit and finishes.
// Measured, cycles at j = 8 (D = 5000 / 46,868): pass A with its loads 3500 / 4000, its exchange 3700 / 8000, pass B 6700 /
// 14500, its exchange 3900 / 6000, pass C 4500 / 11500; the launch 13.6 / 19.9 us on average over a run (23.4 / 26.8 with dots
// split by element, counter barriers and loads where used).  What remains at D = 46,868 is FP64 issue in B and C.
constexpr int OB = 256;   // threads per block of the fused kernel
constexpr long kPollLimit = 1L << 24;        // polls of another block's value (a block may wait for an SM of its own)
constexpr long kBulkLimit = 1L << 20;        // polls of the block's own copies
constexpr int kOrthAlign = 128;              // elements of a block: a multiple of this
constexpr int kOrthSmem = 220 * 1024;        // dynamic shared memory of a block at most
constexpr unsigned long long kEmpty = 0x7ff4dead7ff4deadull;   // a signalling NaN: arithmetic gives quiet ones

// Segmented mode: the vector holds independent problems side by side (a direct sum of superblocks);
// CTA b works on elements [lo_b, hi_b) of segment seg_b, and each segment has its own partial sums,
// tridiagonal (kTriStride doubles), flags (kFlagStride ints) and coefficients (kCoefStride).
constexpr int kTriStride = 128, kFlagStride = 4, kCoefStride = 16 * 32;
struct SegTab {
    const int* cta_seg;
    const int64_t* cta_lo;
    const int64_t* cta_hi;
    const int* seg_cta0;   // first CTA of each segment; seg_cta0[nseg] = the grid
    int nseg;
};

struct OrthArgs {
    const cplx* V;
    cplx* w;
    int64_t n;
    int nv, j, nk;
    double tol;
    double2* partA;    // first-pass partials, rows k of gridDim.x blocks
    double2* partB;    // second-pass partials of this step (empty)
    double2* partC;    // third-pass partials of this step (empty)
    double2 *nextB, *nextC;   // both of the next step (used by the step before): cleared here
    double* tri;
    int* flags;
    int* status;
    int chunk;         // elements of a block (one problem)
    int rows;          // newest Krylov vectors staged in shared memory (STAGED)
    int emax;          // elements of a block at most (shared-memory row)
    SegTab seg;        // seg.nseg == 0: one problem over the whole vector
};

__device__ __forceinline__ double2 ld_slot(const double2* p) {   // two independent 8-byte values
    double2 v;
    asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_slot(double* p, double v) {
    asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ bool is_empty(double v) { return (unsigned long long)__double_as_longlong(v) == kEmpty; }

// h = sum of part[b0 .. b1) in a fixed order (lane l holds blocks b0 + l, b0 + l + 32, ...), waiting for each value; one warp.
// Lanes 0-15 return the real, 16-31 the imaginary part.
__device__ __forceinline__ double poll_sum(const double2* part, int b0, int b1, int* status) {
    constexpr int U = 5;   // values in flight per lane
    const int l = threadIdx.x & 31;
    double re = 0.0, im = 0.0;
    for (int c0 = b0; c0 < b1; c0 += 32 * U) {
        double2 x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = c0 + l + 32 * u < b1 ? ld_slot(part + c0 + l + 32 * u) : make_double2(0.0, 0.0);
        for (long it = 0;; ++it) {   // only what is still empty is read again: all blocks poll the same few lines
            bool ok = true;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (is_empty(x[u].x) || is_empty(x[u].y)) {
                    x[u] = ld_slot(part + c0 + l + 32 * u);
                    ok = false;
                }
            if (__all_sync(0xffffffffu, ok)) break;
            if (it > kPollLimit) {
                if (l == 0) atomicOr(status, 2);
                break;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (c0 + 32 * u >= b1) break;   // uniform: no FP64 instructions for absent values
            re += x[u].x;
            im += x[u].y;
        }
    }
    // lanes 0-15 take the real, 16-31 the imaginary part; then a butterfly over 16 lanes
    const bool up = l & 16;
    double v = (up ? im : re) + __shfl_xor_sync(0xffffffffu, up ? re : im, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// FP32 value of a double by truncating its mantissa to 23 bits, on the integer pipe (conversions and FP64
// arithmetic share this GPU's narrow FP64 pipe); |x| below 2^-126 gives 0.  Relative error <= 2^-23.
__device__ __forceinline__ float f32_trunc(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(b >> 32), ex = (hi >> 20) & 0x7FFu;
    const unsigned mant = ((hi & 0xFFFFFu) << 3) | ((unsigned)b >> 29);
    return ex <= 896u ? 0.f : __uint_as_float((hi & 0x80000000u) | ((ex - 896u) << 23) | mant);
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool wait_bulk(uint32_t bar) {
    for (long i = 0; i < kBulkLimit; ++i) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done) : "r"(bar) : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// <v|x> over one warp's elements (lane, lane + 32, ...) of [0, E)
__device__ __forceinline__ double2 warp_dot(const double2* v, const double2* x, int E) {
    double2 s = make_double2(0.0, 0.0), t = make_double2(0.0, 0.0);
    for (int i = threadIdx.x & 31; i < E; i += 32) {
        const double2 a = v[i], b = x[i];
        s.x = fma(a.x, b.x, s.x);
        t.x = fma(a.y, b.y, t.x);
        s.y = fma(a.x, b.y, s.y);
        t.y = fma(a.y, b.x, t.y);
    }
    return make_double2(s.x + t.x, s.y - t.y);
}

// ||x||^2 over one warp's elements
__device__ __forceinline__ double2 warp_norm2(const double2* x, int E) {
    double s = 0.0, t = 0.0;
    for (int i = threadIdx.x & 31; i < E; i += 32) {
        const double2 v = x[i];
        s = fma(v.x, v.x, s);
        t = fma(v.y, v.y, t);
    }
    return make_double2(s + t, 0.0);
}

// The sum of d over the warp into a slot
__device__ __forceinline__ void store_part(double2* slot, double2 d) {
    const int lane = threadIdx.x & 31;
    const bool up = lane & 16;
    double v = (up ? d.y : d.x) + __shfl_xor_sync(0xffffffffu, up ? d.x : d.y, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 15) == 0) st_slot(reinterpret_cast<double*>(slot) + (lane >> 4), v);
}

// beta, alpha and the stop test of a step from the dots h and the norm h[nv], by one warp; sc = {beta, 1 / beta}, 0 instead
// of 1 / beta to stop and -1 (first: only then) when the pass took more than half of ||w'||^2.
__device__ __forceinline__ void orth_scalars(const OrthArgs& a, double* tri, int* flags, const double2* h, double* alpha1, double* sc,
                                             bool write, bool first) {
    const int lane = threadIdx.x & 31, nv = a.nv;
    double q = lane < nv ? fma(h[lane].x, h[lane].x, h[lane].y * h[lane].y) : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if (lane != 0) return;
    const double bt = sqrt(fmax(h[nv].x - q, 0.0));
    const double alpha = *alpha1 + h[a.j].x;
    const bool st = (a.j == a.nk - 1) || (bt <= a.tol * fmax(1.0, fabs(alpha)));
    // q > ||w'||^2 / 2, by the words that hold the exponents and 20 bits (both are positive)
    const bool again = first && !st && __double2hiint(q) > __double2hiint(h[nv].x) - (1 << 20);
    sc[0] = bt;
    sc[1] = st ? 0.0 : again ? -1.0 : 1.0 / bt;
    if (again) {
        *alpha1 = alpha;
    } else if (write) {
        tri[T_ALPHA + a.j] = alpha;
        tri[T_BETA + a.j] = bt;
        if (st) {
            tri[T_RESID] = bt;
            flags[0] = a.j + 1;   // read by later kernels only (every block is past its check)
        }
    }
}

// The third pass of a step, rare, so it reads V from global memory only: w' - sum h2_k v_k takes the place of w', then (B) and
// (C) with the slots of partC.
__device__ __noinline__ void third_pass(const OrthArgs& a, double* tri, int* flags, const cplx* gV, double2* w, cplx* vnext, double2* h,
                                        double* alpha1, double* sc, int E, int b0, int b1) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nv = a.nv, G = (int)gridDim.x;
    auto update = [&](int i) {
        double2 x = w[i];
        for (int k = 0; k < nv; ++k) {
            const double2 v = gV[(int64_t)k * a.n + i];
            x.x = fma(-h[k].x, v.x, fma(h[k].y, v.y, x.x));
            x.y = fma(-h[k].x, v.y, fma(-h[k].y, v.x, x.y));
        }
        return x;
    };
    for (int i = tid; i < E; i += OB) w[i] = update(i);
    __syncthreads();
    for (int k = warp; k <= nv; k += OB / 32)
        store_part(a.partC + (int64_t)k * G + blockIdx.x, k == nv ? warp_norm2(w, E) : warp_dot(gV + (int64_t)k * a.n, w, E));
    for (int k = warp; k <= nv; k += OB / 32) {
        const double v = poll_sum(a.partC + (int64_t)k * G, b0, b1, a.status);
        if (lane == 0) h[k].x = v;
        if (lane == 16) h[k].y = v;
    }
    __syncthreads();
    if (warp == OB / 32 - 1) orth_scalars(a, tri, flags, h, alpha1, sc, (int)blockIdx.x == b0, false);
    __syncthreads();
    if (sc[1] == 0.0) return;
    for (int i = tid; i < E; i += OB) {
        const double2 x = update(i);
        vnext[i] = make_double2(x.x * sc[1], x.y * sc[1]);
    }
}

template <bool SEG, bool STAGED>
__global__ void __launch_bounds__(OB, 1) k_lanczos_orth_t(const __grid_constant__ OrthArgs a) {
    pdl_enter();
    // one problem: the whole grid stops together.  Segments: nobody waits for a stopped segment's blocks.
    int sg = 0, b0 = 0, b1 = (int)gridDim.x;
    int64_t lo, hi;
    if (SEG) {
        sg = a.seg.cta_seg[blockIdx.x];
        b0 = a.seg.seg_cta0[sg];
        b1 = a.seg.seg_cta0[sg + 1];
        lo = a.seg.cta_lo[blockIdx.x];
        hi = a.seg.cta_hi[blockIdx.x];
    } else {
        lo = min(a.n, (int64_t)blockIdx.x * a.chunk);
        hi = min(a.n, lo + a.chunk);
    }
    double* tri = a.tri + (SEG ? (int64_t)sg * kTriStride : 0);
    int* flags = a.flags + (SEG ? sg * kFlagStride : 0);
    if (a.j >= flags[0]) return;   // stopped (uniform per segment: the flag only changes after the last exchange)
    extern __shared__ double2 osm[];   // STAGED: w, then the newest `rows` Krylov vectors, emax elements each
    __shared__ double2 h[34];
    __shared__ double alpha1, sc[2];
    __shared__ __align__(8) uint64_t bars[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int E = (int)(hi - lo), nv = a.nv, G = (int)gridDim.x;
    const int s0 = STAGED ? nv - a.rows : nv;   // vectors s0 .. nv - 1 are staged
    const cplx* gV = a.V + lo;
    double2* w = STAGED ? osm : a.w + lo;
    auto staged = [&](int k) -> const double2* { return osm + (int64_t)(1 + k - s0) * a.emax; };
    const int j0 = a.j > 0 ? a.j - 1 : 0, na = a.j - j0 + 1;
    if (STAGED) {
        if (tid < 2) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bars + tid)));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0 && E > 0) {   // w, v_{j-1} and v_j first
            const uint32_t bytes = (uint32_t)E * 16u;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bars)), "r"((1 + na) * bytes) : "memory");
            bulk_load(smem_addr(osm), a.w + lo, bytes, smem_addr(bars));
            for (int k = j0; k < nv; ++k) bulk_load(smem_addr(staged(k)), gV + (int64_t)k * a.n, bytes, smem_addr(bars));
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bars + 1)), "r"((j0 - s0) * bytes) : "memory");
            for (int k = s0; k < j0; ++k) bulk_load(smem_addr(staged(k)), gV + (int64_t)k * a.n, bytes, smem_addr(bars + 1));
        }
        if (E > 0 && !wait_bulk(smem_addr(bars))) atomicOr(a.status, 2);
    }
    // (A) first-pass dots (FP32, summed in FP64 from the warps on) with v_{j-1} and v_j only: H v_j has components
    // above rounding along these two alone (the three-term recurrence), so the first pass skips the older vectors
    const double2* v0 = STAGED ? staged(j0) : gV + (int64_t)j0 * a.n;
    const double2* v1 = STAGED ? staged(a.j) : gV + (int64_t)a.j * a.n;
    {
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i = tid; i < E; i += OB) {
            const double2 x = w[i], p = v0[i], q = v1[i];
            const float xr = f32_trunc(x.x), xi = f32_trunc(x.y);
            const float pr = f32_trunc(p.x), pi = f32_trunc(p.y), qr = f32_trunc(q.x), qi = f32_trunc(q.y);
            f.x = fmaf(pr, xr, fmaf(pi, xi, f.x));
            f.y = fmaf(pr, xi, fmaf(-pi, xr, f.y));
            f.z = fmaf(qr, xr, fmaf(qi, xi, f.z));
            f.w = fmaf(qr, xi, fmaf(-qi, xr, f.w));
        }
        double r = 0.0;   // lane l ends with component l / 8 of the warp's sums
        if (warp * 32 < E) {
            const bool u16 = lane & 16, u8 = lane & 8;
            double k0 = u16 ? (double)f.z : (double)f.x, k1 = u16 ? (double)f.w : (double)f.y;
            k0 += __shfl_xor_sync(0xffffffffu, u16 ? (double)f.x : (double)f.z, 16);
            k1 += __shfl_xor_sync(0xffffffffu, u16 ? (double)f.y : (double)f.w, 16);
            r = (u8 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, u8 ? k0 : k1, 8);
            r += __shfl_xor_sync(0xffffffffu, r, 4);
            r += __shfl_xor_sync(0xffffffffu, r, 2);
            r += __shfl_xor_sync(0xffffffffu, r, 1);
        }
        double* shd = reinterpret_cast<double*>(h);   // [component][warp]
        if ((lane & 7) == 0) shd[(lane >> 3) * 8 + warp] = r;
        __syncthreads();
        if (warp == 0) {   // lane = 8 component + warp
            double t = shd[lane];
            t += __shfl_xor_sync(0xffffffffu, t, 4);
            t += __shfl_xor_sync(0xffffffffu, t, 2);
            t += __shfl_xor_sync(0xffffffffu, t, 1);
            // components 0, 1: v_{j-1}; 2, 3: v_j (row na - 1; with j = 0 both are v_0, stored once)
            const int row = na == 2 ? lane >> 4 : 0;
            if ((lane & 7) == 0 && (na == 2 || lane >= 16))
                st_slot(reinterpret_cast<double*>(a.partA + (int64_t)row * G + blockIdx.x) + ((lane >> 3) & 1), t);
        }
    }
    __syncthreads();
    if (warp < na) {
        const double v = poll_sum(a.partA + (int64_t)warp * G, b0, b1, a.status);
        if (lane == 0) h[warp].x = v;
        if (lane == 16) h[warp].y = v;
    }
    __syncthreads();
    // (B) w' = w - h1_{j-1} v_{j-1} - h1_j v_j
    {
        const double2 p = h[0], q = na == 2 ? h[1] : make_double2(0.0, 0.0);
        if (tid == 0) alpha1 = h[na - 1].x;
        for (int i = tid; i < E; i += OB) {
            double2 x = w[i];
            const double2 u = v0[i];
            x.x = fma(-p.x, u.x, fma(p.y, u.y, x.x));
            x.y = fma(-p.x, u.y, fma(-p.y, u.x, x.y));
            if (na == 2) {
                const double2 v = v1[i];
                x.x = fma(-q.x, v.x, fma(q.y, v.y, x.x));
                x.y = fma(-q.x, v.y, fma(-q.y, v.x, x.y));
            }
            w[i] = x;
        }
    }
    if (STAGED && E > 0 && !wait_bulk(smem_addr(bars + 1))) atomicOr(a.status, 2);
    __syncthreads();
    // second-pass dots with every v_k and ||w'||^2 (row nv), FP64: a warp per row
    for (int k = warp; k <= nv; k += OB / 32) {
        const double2 d = k == nv ? warp_norm2(w, E) : STAGED && k >= s0 ? warp_dot(staged(k), osm, E) : warp_dot(gV + (int64_t)k * a.n, w, E);
        store_part(a.partB + (int64_t)k * G + blockIdx.x, d);
    }
    for (int k = warp; k <= nv; k += OB / 32) {
        const double v = poll_sum(a.partB + (int64_t)k * G, b0, b1, a.status);
        if (lane == 0) h[k].x = v;
        if (lane == 16) h[k].y = v;
    }
    // every block of the problem has stored its second-pass partials, so it has read the first-pass ones, and the step
    // before has ended: its own slots of these are cleared for the next step
    __syncthreads();
    {
        const double e = __longlong_as_double((long long)kEmpty);
        if (tid < 2 * na) st_slot(reinterpret_cast<double*>(a.partA + (int64_t)(tid >> 1) * G + blockIdx.x) + (tid & 1), e);
        if (tid < 2 * (nv + 1)) {
            st_slot(reinterpret_cast<double*>(a.nextB + (int64_t)(tid >> 1) * G + blockIdx.x) + (tid & 1), e);
            st_slot(reinterpret_cast<double*>(a.nextC + (int64_t)(tid >> 1) * G + blockIdx.x) + (tid & 1), e);
        }
    }
    // (C) beta, stop test and 1 / beta by the last warp (h2 in parallel, one FP64 square root), beside the others'
    // update x = w' - sum h2_k v_k
    if (warp == OB / 32 - 1) orth_scalars(a, tri, flags, h, &alpha1, sc, (int)blockIdx.x == b0, true);
    const bool last_step = a.j == a.nk - 1;   // no next vector
    cplx* vnext = const_cast<cplx*>(a.V) + (int64_t)(a.j + 1) * a.n + lo;
    bool have_sc = false;
    for (int i0 = 0; i0 < E && !last_step; i0 += OB) {
        const int i = i0 + tid;
        double2 x = make_double2(0.0, 0.0);
        if (i < E) {
            x = w[i];
            int k = 0;
            for (; k + 4 <= s0; k += 4) {   // not staged: four loads in flight
                double2 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = gV[(int64_t)(k + u) * a.n + i];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    x.x = fma(-h[k + u].x, v[u].x, fma(h[k + u].y, v[u].y, x.x));
                    x.y = fma(-h[k + u].x, v[u].y, fma(-h[k + u].y, v[u].x, x.y));
                }
            }
            for (; k < s0; ++k) {
                const double2 v = gV[(int64_t)k * a.n + i];
                x.x = fma(-h[k].x, v.x, fma(h[k].y, v.y, x.x));
                x.y = fma(-h[k].x, v.y, fma(-h[k].y, v.x, x.y));
            }
            if (STAGED)
#pragma unroll 4
                for (; k < nv; ++k) {
                    const double2 v = staged(k)[i];
                    x.x = fma(-h[k].x, v.x, fma(h[k].y, v.y, x.x));
                    x.y = fma(-h[k].x, v.y, fma(-h[k].y, v.x, x.y));
                }
        }
        if (!have_sc) { __syncthreads(); have_sc = true; }   // sc
        if (!(sc[1] > 0.0)) break;   // stopped, or another pass
        if (i < E) vnext[i] = make_double2(x.x * sc[1], x.y * sc[1]);
    }
    if (last_step) return;
    if (!have_sc) __syncthreads();   // a block without elements
    if (sc[1] < 0.0) third_pass(a, tri, flags, gV, w, vnext, h, &alpha1, sc, E, b0, b1);
}

// Taylor terms for a substep with ||T h|| <= xs <= 2: the smallest K (per bucket of xs) whose remainder
// bound xs^{K+1} / (K+1)! is below 1e-17.
__device__ __forceinline__ int taylor_terms(double xs) {
    return xs <= 0.25 ? 12 : xs <= 0.5 ? 15 : xs <= 0.75 ? 17 : xs <= 1.0 ? 18 : xs <= 1.25 ? 20 : xs <= 1.5 ? 21
         : xs <= 1.75 ? 23 : 24;
}

struct Times { double t[16]; };

// Order key of a time t >= 0: unsigned comparison of the bits is numeric comparison (-0 taken as +0).
__device__ __forceinline__ unsigned long long time_key(double v) {
    return (unsigned long long)__double_as_longlong(v == 0.0 ? 0.0 : v);
}

// 1/k for the Taylor terms (k <= 24), correctly rounded at compile time.
__constant__ double kInvK[25] = {0.0, 1.0 / 1, 1.0 / 2, 1.0 / 3, 1.0 / 4, 1.0 / 5, 1.0 / 6, 1.0 / 7, 1.0 / 8,
                                 1.0 / 9, 1.0 / 10, 1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16,
                                 1.0 / 17, 1.0 / 18, 1.0 / 19, 1.0 / 20, 1.0 / 21, 1.0 / 22, 1.0 / 23, 1.0 / 24};

// c_x = beta0 e^{-i T t_x} e_0 for the Lanczos tridiagonal T (alpha, beta), the quantity of
// Eq. lanczosevolution (there written through T = S^dag D S).  GB300 has little FP64 throughput per
// SM, and a Jacobi diagonalisation in one warp spends thousands of dependent FP64 instructions, so
// the vector is advanced directly: one lane per component, (T u)_l from the neighbours by shuffles,
// Taylor series on substeps h with ||T h|| <= nu |h| <= 2 (nu the Gershgorin bound), 12-24 terms
// chosen so that the remainder (nu |h|)^{K+1} / (K+1)! stays below 1e-17.  Targets are reached in
// order of time from t = 0, each from the previous one.  The Krylov error estimate is
// beta_n beta0 |[e^{-i T t_max} e_0]_{n-1}| (t_max the largest target time).
__global__ void __launch_bounds__(32) k_tridiag_exp(double* __restrict__ tri, const int* __restrict__ flags,
                                                     Times times, int n_v, cplx* __restrict__ coef) {
    pdl_enter();
    // one block per segment in segmented mode (a single block otherwise)
    tri += (int64_t)blockIdx.x * kTriStride;
    flags += blockIdx.x * kFlagStride;
    coef += (int64_t)blockIdx.x * kCoefStride;
    __shared__ int order[16];
    const int l = threadIdx.x;
    const int n = flags[0];
    const double b0 = tri[T_BETA0];
    for (int x = 0; x < n_v; ++x) coef[x * 32 + l] = make_double2(0.0, 0.0);
    if (n <= 0) {
        if (l == 0) tri[T_ERR] = 0.0;
        return;
    }
    const double al = l < n ? tri[T_ALPHA + l] : 0.0;
    const double bl = l < n - 1 ? tri[T_BETA + l] : 0.0;   // couples l and l + 1
    double bm = __shfl_up_sync(0xffffffffu, bl, 1);        // couples l - 1 and l
    if (l == 0) bm = 0.0;
    double nu = fabs(al) + fabs(bl) + fabs(bm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nu = fmax(nu, __shfl_xor_sync(0xffffffffu, nu, o));
    if (l == 0) {   // targets by increasing time
        unsigned long long key[16];
        for (int x = 0; x < n_v; ++x) { key[x] = time_key(times.t[x]); order[x] = x; }
        for (int x = 1; x < n_v; ++x)
            for (int y = x; y > 0 && key[order[y - 1]] > key[order[y]]; --y) { const int t = order[y]; order[y] = order[y - 1]; order[y - 1] = t; }
    }
    __syncwarp();
    int xmax = 0;
    double tmax = 0.0;
    for (int x = 0; x < n_v; ++x)
        if (times.t[x] > tmax) { tmax = times.t[x]; xmax = x; }
    // t_x >= 0 (checked by the entry point): each target from the previous one in time order
    double2 u0 = make_double2(l == 0 ? 1.0 : 0.0, 0.0);   // e^{-i T t_prev} e_0
    double tprev = 0.0;
    for (int m = 0; m < n_v; ++m) {
        const int x = order[m];
        const double dt = times.t[x] - tprev;
        const double span = nu * dt;
        const int S = span > 0.0 ? (int)ceil(0.5 * span) : 0;
        if (S > 0) {
            const double h = dt / S, xs = nu * h;
            const int K = taylor_terms(xs);
            for (int st = 0; st < S; ++st) {
                double2 u = u0, sum = u0;
                for (int k = 1; k <= K; ++k) {
                    const double lx = __shfl_up_sync(0xffffffffu, u.x, 1), ly = __shfl_up_sync(0xffffffffu, u.y, 1);
                    const double rx = __shfl_down_sync(0xffffffffu, u.x, 1), ry = __shfl_down_sync(0xffffffffu, u.y, 1);
                    const double tx = fma(bl, rx, fma(bm, lx, al * u.x));   // (T u)_l; bm = 0 on lane 0,
                    const double ty = fma(bl, ry, fma(bm, ly, al * u.y));   // bl = 0 from lane n - 1 on
                    const double f = h * kInvK[k];
                    u = make_double2(f * ty, -f * tx);                      // (-i h / k) T u
                    sum.x += u.x; sum.y += u.y;
                }
                u0 = sum;
            }
        }
        tprev = times.t[x];
        if (l < n) coef[x * 32 + l] = make_double2(b0 * u0.x, b0 * u0.y);
        if (x == xmax && l == n - 1) tri[T_ERR] = tri[T_RESID] * b0 * sqrt(u0.x * u0.x + u0.y * u0.y);
    }
}

// Targets at equally spaced times m dt (m = 0 .. n_v - 1, target order[m] at m dt): the same c_x as
// k_tridiag_exp, with the chain of dependent Taylor terms one time step long instead of n_v - 1.  Block c
// forms column c of the step exponential E = e^{-i T dt} (the Taylor substeps of k_tridiag_exp from e_c,
// lane l = row l); the last block to finish (ticket) takes u_0 = e_0, u_m = E u_{m-1}.
struct StepTimes { double dt; int n_v, xmax; int order[16]; };
__global__ void __launch_bounds__(32) k_tridiag_exp_eq(double* __restrict__ tri, const int* __restrict__ flags,
                                                        StepTimes st, cplx* __restrict__ coef, cplx* __restrict__ mexp,
                                                        unsigned* __restrict__ ticket) {
    pdl_enter();
    const int l = threadIdx.x, c = blockIdx.x;
    const int n = flags[0];
    if (c < n) {
        const double al = l < n ? tri[T_ALPHA + l] : 0.0;
        const double bl = l < n - 1 ? tri[T_BETA + l] : 0.0;   // couples l and l + 1
        double bm = __shfl_up_sync(0xffffffffu, bl, 1);        // couples l - 1 and l
        if (l == 0) bm = 0.0;
        double nu = fabs(al) + fabs(bl) + fabs(bm);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nu = fmax(nu, __shfl_xor_sync(0xffffffffu, nu, o));
        double2 u0 = make_double2(l == c ? 1.0 : 0.0, 0.0);
        const double span = nu * st.dt;
        const int S = span > 0.0 ? (int)ceil(0.5 * span) : 0;
        if (S > 0) {
            const double h = st.dt / S, xs = nu * h;
            const int K = taylor_terms(xs);
            for (int sb = 0; sb < S; ++sb) {
                double2 u = u0, sum = u0;
                for (int k = 1; k <= K; ++k) {
                    const double lx = __shfl_up_sync(0xffffffffu, u.x, 1), ly = __shfl_up_sync(0xffffffffu, u.y, 1);
                    const double rx = __shfl_down_sync(0xffffffffu, u.x, 1), ry = __shfl_down_sync(0xffffffffu, u.y, 1);
                    const double tx = fma(bl, rx, fma(bm, lx, al * u.x));
                    const double ty = fma(bl, ry, fma(bm, ly, al * u.y));
                    const double f = h * kInvK[k];
                    u = make_double2(f * ty, -f * tx);                      // (-i h / k) T u
                    sum.x += u.x; sum.y += u.y;
                }
                u0 = sum;
            }
        }
        mexp[c * 32 + l] = u0;
    }
    __threadfence();
    unsigned tk = 0;
    if (l == 0) tk = atomicAdd(ticket, 1u);
    tk = __shfl_sync(0xffffffffu, tk, 0);
    if (tk != gridDim.x - 1) return;   // not the last block
    __threadfence();
    if (l == 0) *ticket = 0u;          // every block has taken its ticket: ready for the next launch
    const double b0 = tri[T_BETA0];
    for (int x = 0; x < st.n_v; ++x) coef[x * 32 + l] = make_double2(0.0, 0.0);
    if (n <= 0) {
        if (l == 0) tri[T_ERR] = 0.0;
        return;
    }
    double2 u = make_double2(l == 0 ? 1.0 : 0.0, 0.0);
    for (int m = 0; m < st.n_v; ++m) {
        if (m > 0) {   // u <- E u, two partial sums
            double2 a0 = make_double2(0.0, 0.0), a1 = make_double2(0.0, 0.0);
            for (int cc = 0; cc < n; cc += 2) {   // lanes >= n hold u = 0, so column n (if n is odd) adds 0
                const double ux = __shfl_sync(0xffffffffu, u.x, cc), uy = __shfl_sync(0xffffffffu, u.y, cc);
                const double vx = __shfl_sync(0xffffffffu, u.x, cc + 1), vy = __shfl_sync(0xffffffffu, u.y, cc + 1);
                const double2 e = __ldcg(mexp + cc * 32 + l);
                const double2 f = cc + 1 < n ? __ldcg(mexp + (cc + 1) * 32 + l) : make_double2(0.0, 0.0);
                a0.x = fma(e.x, ux, fma(-e.y, uy, a0.x));
                a0.y = fma(e.x, uy, fma(e.y, ux, a0.y));
                a1.x = fma(f.x, vx, fma(-f.y, vy, a1.x));
                a1.y = fma(f.x, vy, fma(f.y, vx, a1.y));
            }
            u = make_double2(a0.x + a1.x, a0.y + a1.y);
        }
        const int x = st.order[m];
        if (l < n) coef[x * 32 + l] = make_double2(b0 * u.x, b0 * u.y);
        if (x == st.xmax && l == n - 1) tri[T_ERR] = tri[T_RESID] * b0 * sqrt(u.x * u.x + u.y * u.y);
    }
}

// The pair times one power of two, by integer instructions (the FP64 pipe is what bounds the chains below): the larger
// between 1/2 and 1, a zero or what falls below 2^-1022 gives 0.
__device__ __forceinline__ void rescale_pair(double& x, double& y) {
    const int hx = __double2hiint(x), hy = __double2hiint(y);
    const int ex = (hx >> 20) & 0x7FF, ey = (hy >> 20) & 0x7FF, s = 1022 - max(ex, ey);
    x = ex == 0 || ex + s <= 0 ? 0.0 : __hiloint2double(hx + (s << 20), __double2loint(x));
    y = ey == 0 || ey + s <= 0 ? 0.0 : __hiloint2double(hy + (s << 20), __double2loint(y));
}

// Lowest eigenpair of the Lanczos tridiagonal T (ground-state targeting, Sec. II.B), FP64, n <= 32.
// The eigenvalue by multisection: x lies below it exactly when the leading minors d_k = det(T_k - x) are all
// positive, d_k = (alpha_k - x) d_{k-1} - beta_{k-1}^2 d_{k-2} with T scaled by a power of two to norm <= 1.
// 128 threads try 128 points of the bracket at once, so it shrinks 129-fold in one chain of n steps.  Only the signs
// count, so the pair (d_{k-1}, d_k) is scaled by a power of two every four steps: without it the minors of a T whose
// spread is small against its norm (a constant or a penalty in H) underflow from ||T|| / 1e10 on, and the bracket walks
// to an end of the Gershgorin interval.
// Then the eigenvalue is known to 4e-16 of its size, which may be as much as the distance to the next.  The rest works on
// T - lambda, whose differences are rounded relative to themselves: where the spread of T about lambda calls for it, the
// bracket around 0 is narrowed to 4e-15 of that spread (no step for an ordinary spectrum).
// The eigenvector by the twisted factorisation of T - lambda (Dhillon 1997): pivots p_k from the top and m_k from the
// bottom (ratios of neighbouring leading and trailing minors), the twist r where |p_k + m_k - (alpha_k - lambda)| is
// smallest, z_r = 1, z_k = -(beta_k / p_k) z_{k+1} above and z_k = -(beta_{k-1} / m_k) z_{k-1} below: one lane per
// component, products by scans.  A pivot below eps |lambda| (a leading or trailing block with the same eigenvalue, or n = 1)
// is replaced by that, in the minor itself, so that the pivots after it follow.  coef[0][k] = z_k / |z| (real),
// tri[T_EMIN] = lambda.  ~30 us at n = 32, bound by the FP64 pipe: three instructions of 64 cycles a step and warp.
constexpr int kMinThreads = 128;
__global__ void __launch_bounds__(kMinThreads) k_tridiag_min(double* __restrict__ tri, const int* __restrict__ flags,
                                                              cplx* __restrict__ coef) {
    pdl_enter();
    const int n = flags[0], tid = threadIdx.x, l = tid & 31;
    if (tid < 32) coef[tid] = make_double2(0.0, 0.0);
    if (n <= 0) {
        if (tid == 0) tri[T_EMIN] = 0.0;
        return;
    }
    __shared__ double sa[32], sb2[32], sx[kMinThreads + 2], sd[2][32], sq[2][32];
    // every warp: alpha_l, beta_l (couples l and l + 1) and the Gershgorin interval
    double al = l < n ? tri[T_ALPHA + l] : 0.0, be = l < n - 1 ? tri[T_BETA + l] : 0.0;
    double bm = __shfl_up_sync(0xffffffffu, be, 1);
    if (l == 0) bm = 0.0;
    const double r = fabs(be) + fabs(bm);
    double lo = l < n ? al - r : 1e300, hi = l < n ? al + r : -1e300;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const double nrm = fmax(fabs(lo), fabs(hi));
    int e2 = 0;
    frexp(nrm, &e2);
    e2 = max(e2, -1000);   // 2^-e2 stays finite
    const double sc = nrm > 0.0 ? ldexp(1.0, -e2) : 1.0, us = nrm > 0.0 ? ldexp(1.0, e2) : 1.0;
    al *= sc; be *= sc; bm *= sc; lo *= sc; hi *= sc;
    if (tid < 32) { sa[l] = al; sb2[l] = be * be; }
    __syncthreads();
    auto narrow = [&]() {   // the bracket [lo, hi] shrinks 129-fold
        const double x = fma(hi - lo, (tid + 1) * (1.0 / (kMinThreads + 1)), lo);
        double d0 = 1.0, d1 = sa[0] - x;
        bool below = d1 > 0.0;
        for (int k = 1; k < n; ++k) {
            const double d2 = fma(sa[k] - x, d1, -sb2[k - 1] * d0);
            d0 = d1;
            d1 = d2;
            below = below && d2 > 0.0;
            if ((k & 3) == 0) rescale_pair(d0, d1);
        }
        sx[tid + 1] = x;
        if (tid == 0) { sx[0] = lo; sx[kMinThreads + 1] = hi; }
        const int c = __syncthreads_count(below);   // points below the eigenvalue: the first c of them
        lo = sx[c];
        hi = sx[c + 1];
        __syncthreads();
    };
    for (int it = 0; it < 28 && hi - lo > 4e-16 * fmax(fabs(lo), fabs(hi)) + 1e-300; ++it) narrow();
    // T - base from here on; the counts so far are exact for entries off by a few eps of the spread
    const double base = 0.5 * (lo + hi);
    al -= base;
    double sp = l < n ? fabs(al) + fabs(be) + fabs(bm) : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sp = fmax(sp, __shfl_xor_sync(0xffffffffu, sp, o));
    if (tid < 32) sa[l] = al;
    lo = lo - base - 1e-15 * sp;
    hi = hi - base + 1e-15 * sp;
    __syncthreads();
    for (int it = 0; it < 12 && hi - lo > 4e-15 * sp; ++it) narrow();
    if (tid >= 32) return;
    const double lam = 0.5 * (lo + hi);
    al -= lam;
    sa[l] = al;
    __syncwarp();
    const double pmin = fmax(2.2e-16 * fabs(base + lam), 0x1p-200);
    if (l < 2) {   // lane 0: leading minors, lane 1: trailing minors of T - lambda, each with the one before it
        double d0 = 0.0, d1 = 1.0, b2 = 0.0;
        for (int k = 0; k < n; ++k) {
            const int i = l == 0 ? k : n - 1 - k;
            double d2 = fma(sa[i], d1, -b2 * d0);
            const double lim = pmin * d1;
            if (!(fabs(d2) >= fabs(lim))) d2 = copysign(lim, d2);
            sd[l][i] = d2;
            sq[l][i] = d1;
            d0 = d1;
            d1 = d2;
            b2 = l == 0 ? sb2[i] : (i > 0 ? sb2[i - 1] : 0.0);
            if ((k & 3) == 3) rescale_pair(d0, d1);
        }
    }
    __syncwarp();
    const bool in = l < n;
    const double p = in ? sd[0][l] / sq[0][l] : 1.0;
    const double m = in ? sd[1][l] / sq[1][l] : 1.0;
    double g = in ? fabs(p + m - al) : 1e300;
    int tw = l;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {   // the smallest, ties to the first
        const double og = __shfl_xor_sync(0xffffffffu, g, o);
        const int ot = __shfl_xor_sync(0xffffffffu, tw, o);
        if (og < g || (og == g && ot < tw)) { g = og; tw = ot; }
    }
    double up = l < tw ? -be / p : 1.0;                 // z_l = product of up over l .. tw - 1
    double dn = in && l > tw ? -bm / m : 1.0;           // z_l = product of dn over tw + 1 .. l
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_down_sync(0xffffffffu, up, o), d = __shfl_up_sync(0xffffffffu, dn, o);
        if (l + o < 32) up *= u;
        if (l >= o) dn *= d;
    }
    const double z = in ? (l < tw ? up : dn) : 0.0;
    double mx = fabs(z);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const double zs = z / mx;   // mx >= |z_tw| = 1
    double nn = zs * zs;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
    if (in) coef[l] = make_double2(zs / sqrt(nn), 0.0);
    if (l == 0) tri[T_EMIN] = (base + lam) * us;
}

struct TargetPtrs { cplx* p[16]; };
struct CombineList { cplx* p[16]; int row[16]; int n; };   // targets and their coefficient rows

// sum_k c[k] v_k[i] over nu vectors, four loads ahead of their use
__device__ __forceinline__ double2 combine_one(const cplx* __restrict__ V, int64_t n, int64_t i, const double2* c, int nu) {
    double2 acc = make_double2(0.0, 0.0);
    auto add = [&](double2 w, double2 v) {
        acc.x = fma(w.x, v.x, fma(-w.y, v.y, acc.x));
        acc.y = fma(w.x, v.y, fma(w.y, v.x, acc.y));
    };
    int k = 0;
    for (; k + 4 <= nu; k += 4) {
        double2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = V[(int64_t)(k + u) * n + i];
#pragma unroll
        for (int u = 0; u < 4; ++u) add(c[k + u], v[u]);
    }
    for (; k < nu; ++k) add(c[k], V[(int64_t)k * n + i]);
    return acc;
}

// targets p[x][i] = sum_k coef[row[x]][k] v_k[i], one target per blockIdx.y.  What bounds it is FP64 issue (4 instructions
// of 64 cycles per k and element), so what counts is that every sub-partition has work and an even share: with all targets
// in one thread's registers and V read once, 5332 elements kept 167 of 608 sub-partitions busy for 9200 cycles and loads
// came one at a time.  The second and third read of V come from L2.  Measured with n_K = 12 and three targets at
// D = 5332, n_K = 10 at D = 46,868: the whole advance 417.7 -> 410.9 us and 679.0 -> 674.4 us.
constexpr int CBT = 128;
__global__ void __launch_bounds__(CBT) k_combine(const cplx* __restrict__ V, int64_t n, const int* __restrict__ flags,
                                                 const cplx* __restrict__ coef, CombineList tg) {
    pdl_enter();
    __shared__ double2 cf[32];
    const int nu = flags[0], x = blockIdx.y;
    if (threadIdx.x < 32) cf[threadIdx.x] = coef[tg.row[x] * 32 + threadIdx.x];
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * CBT + threadIdx.x; i < n; i += (int64_t)gridDim.x * CBT) tg.p[x][i] = combine_one(V, n, i, cf, nu);
}

// The targets listed in rows (coefficient row of each).  Of segmented targets in one buffer the last is formed, as the
// blocks of different targets run in any order.
CombineList combine_list(const std::vector<int>& rows, const TargetPtrs& tg) {
    CombineList t{};
    for (size_t x = 0; x < rows.size(); ++x) {
        bool again = false;
        for (size_t y = x + 1; y < rows.size(); ++y) again |= tg.p[rows[y]] == tg.p[rows[x]];
        if (again) continue;
        t.p[t.n] = tg.p[rows[x]];
        t.row[t.n++] = rows[x];
    }
    return t;
}
int launch_combine(const cplx* V, int64_t n, const int* flags, const cplx* coef, const std::vector<int>& rows,
                   const TargetPtrs& tg, int sms, cudaStream_t s) {
    const CombineList t = combine_list(rows, tg);
    if (t.n == 0) return 0;
    const int grid = (int)std::min<int64_t>((n + CBT - 1) / CBT, 16L * sms);
    launch_pdl(k_combine, dim3(grid, t.n), CBT, 0, s, V, n, flags, coef, t);
    return 1;
}

// ---- segmented mode: the start vector's norm, v_0 and the targets per segment --------------------
__global__ void __launch_bounds__(NT) k_norm2_seg(const cplx* __restrict__ x, SegTab tb, double2* __restrict__ part) {
    pdl_enter();
    const int64_t lo = tb.cta_lo[blockIdx.x], hi = tb.cta_hi[blockIdx.x];
    double s = 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += NT) { const double2 v = x[i]; s += v.x * v.x + v.y * v.y; }
    const double2 t = block_sum(make_double2(s, 0.0));
    if (threadIdx.x == 0) part[blockIdx.x] = t;
}

__global__ void __launch_bounds__(NT) k_init_v0_seg(const cplx* __restrict__ phi, SegTab tb, const double2* __restrict__ part,
                                                    cplx* __restrict__ v0, double* __restrict__ tri, int* __restrict__ flags,
                                                    int nk, OrthSlots slots) {
    pdl_enter();
    clear_slots(slots);
    __shared__ double sb[2];
    const int sg = tb.cta_seg[blockIdx.x], c0 = tb.seg_cta0[sg], c1 = tb.seg_cta0[sg + 1];
    if (threadIdx.x < 32) {   // the segment's partials in a fixed order
        double t = 0.0;
        for (int b = c0 + (int)threadIdx.x; b < c1; b += 32) t += part[b].x;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) {
            sb[0] = sqrt(t);
            sb[1] = sb[0] > 0.0 ? 1.0 / sb[0] : 0.0;
        }
    }
    __syncthreads();
    const double b0 = sb[0], inv = sb[1];
    const int64_t lo = tb.cta_lo[blockIdx.x], hi = tb.cta_hi[blockIdx.x];
    for (int64_t i = lo + threadIdx.x; i < hi; i += NT) { const double2 v = phi[i]; v0[i] = make_double2(v.x * inv, v.y * inv); }
    if ((int)blockIdx.x == c0 && threadIdx.x == 0) {
        tri[(int64_t)sg * kTriStride + T_BETA0] = b0;
        tri[(int64_t)sg * kTriStride + T_RESID] = 0.0;
        flags[sg * kFlagStride] = b0 > 0.0 ? nk : 0;
    }
}

// The targets over each block's range with its segment's coefficients, one target per blockIdx.y
__global__ void __launch_bounds__(CBT) k_combine_seg(const cplx* __restrict__ V, int64_t n, SegTab tb, const int* __restrict__ flags,
                                                     const cplx* __restrict__ coef, CombineList tg) {
    pdl_enter();
    __shared__ double2 cf[32];
    const int sg = tb.cta_seg[blockIdx.x], nu = flags[sg * kFlagStride], x = blockIdx.y;
    if (threadIdx.x < 32) cf[threadIdx.x] = coef[(int64_t)sg * kCoefStride + tg.row[x] * 32 + threadIdx.x];
    __syncthreads();
    const int64_t lo = tb.cta_lo[blockIdx.x], hi = tb.cta_hi[blockIdx.x];
    for (int64_t i = lo + threadIdx.x; i < hi; i += CBT) tg.p[x][i] = combine_one(V, n, i, cf, nu);
}

__global__ void __launch_bounds__(NT) k_dot2(const cplx* __restrict__ x, const cplx* __restrict__ y, int64_t n,
                                              double2* __restrict__ part) {
    pdl_enter();
    int64_t lo, hi;
    chunk_of(n, lo, hi);
    double2 s = make_double2(0.0, 0.0);
    double nn = 0.0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += NT) {
        const double2 a = x[i];
        const double2 p = cdotc(a, y[i]);
        s.x += p.x; s.y += p.y;
        nn += a.x * a.x + a.y * a.y;
    }
    double2 t = block_sum(s);
    double2 u = block_sum(make_double2(nn, 0.0));
    if (threadIdx.x == 0) { part[blockIdx.x] = t; part[NB + blockIdx.x] = u; }
}

__global__ void __launch_bounds__(NT) k_dot_final(const double2* __restrict__ part, cplx* __restrict__ out, int normalise) {
    pdl_enter();
    __shared__ double2 h[2];
    reduce_coeffs(part, 2, h);
    if (threadIdx.x == 0) {
        double2 v = h[0];
        if (normalise) {
            const double d = h[1].x > 0.0 ? 1.0 / h[1].x : 0.0;
            v.x *= d; v.y *= d;
        }
        *out = v;
    }
}

int ensure_work(tdmrg_ctx* c, int a, int b, int nk, int64_t n, KrylovWork** out) {
    auto key = std::make_pair(a * 4096 + b, nk);
    auto it = c->krylov.find(key);
    if (it != c->krylov.end() && it->second.n == n) { *out = &it->second; return TDMRG_OK; }
    KrylovWork k;
    k.n = n;
    k.nk = nk;
    int rc = dev_alloc(c, (void**)&k.V, (size_t)(nk + 1) * n * sizeof(cplx), "Krylov vectors");
    if (!rc) rc = dev_alloc(c, (void**)&k.w, (size_t)n * sizeof(cplx), "Krylov residual");
    if (!rc) rc = dev_alloc(c, (void**)&k.part, part_bytes(nk), "Krylov partials");
    if (!rc) rc = dev_alloc(c, (void**)&k.tri, 128 * sizeof(double), "Krylov tridiagonal");
    if (!rc) rc = dev_alloc(c, (void**)&k.flags, 4 * sizeof(int), "Krylov flags");
    // coefficients [x][k] of 16 targets, then the columns of the step exponential (32 x 32)
    if (!rc) rc = dev_alloc(c, (void**)&k.coef, kCoefWords * sizeof(cplx), "Krylov coefficients");
    // the ticket of k_tridiag_exp_eq (word 2)
    if (!rc) rc = dev_alloc(c, (void**)&k.bar, kBarWords * sizeof(unsigned), "Krylov ticket");
    if (!rc) rc = cuda_check(c, cudaMemsetAsync(k.bar, 0, kBarWords * sizeof(unsigned), c->stream), "Krylov ticket");
    if (!rc) {   // co-resident grid of the fused orthogonalisation: at most one block per SM, at most NB
        int per_sm = 0;
        rc = cuda_check(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lanczos_orth_t<true, false>, OB, 0), "occupancy");
        const int want = c->orth_per_sm > 0 ? c->orth_per_sm : 1;   // blocks per SM of the fused orthogonalisation
        k.orth_per_sm = std::max(1, std::min(want, std::max(per_sm, 1)));
        k.orth_grid = std::max(1, std::min(c->num_sms * k.orth_per_sm, NB));
        // the opt-in is a property of the kernels on the device: always the maximum
        for (const void* f : {(const void*)k_lanczos_orth_t<false, true>, (const void*)k_lanczos_orth_t<true, true>})
            if (!rc) rc = cuda_check(c, cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kOrthSmem), "orthogonalisation smem");
    }
    if (rc) {
        dev_free(c, k.V, (size_t)(nk + 1) * n * sizeof(cplx));
        dev_free(c, k.w, (size_t)n * sizeof(cplx));
        dev_free(c, k.part, part_bytes(nk));
        dev_free(c, k.tri, 128 * sizeof(double));
        dev_free(c, k.flags, 4 * sizeof(int));
        dev_free(c, k.coef, kCoefWords * sizeof(cplx));
        dev_free(c, k.bar, kBarWords * sizeof(unsigned));
        return rc;
    }
    c->krylov[key] = k;
    *out = &c->krylov[key];
    return TDMRG_OK;
}

}  // namespace

cudaError_t launch_dot_final(const cplx* x, const cplx* y, int64_t n, double2* partials, int nblk, cplx* out,
                             int normalise, cudaStream_t s) {
    (void)nblk;
    launch_pdl(k_dot2, NB, NT, 0, s, x, y, n, partials);
    launch_pdl(k_dot_final, 1, NT, 0, s, partials, out, normalise);
    return cudaGetLastError();
}

// Partial-sum slots of a Lanczos run on `grid` blocks with nk steps; norm partials of the start vector are in row 2.
static OrthSlots orth_slots(const KrylovWork* k, int grid, int nk) {
    const int64_t buf = (nk + 1) * (int64_t)kRedBlocks;
    double2* const b = k->part + 3 * (int64_t)kRedBlocks;
    return OrthSlots{k->part, {b, b + buf}, {b + 2 * buf, b + 3 * buf}, nk + 1, grid};
}
static double2* norm_slots(const KrylovWork* k) { return k->part + 2 * (int64_t)kRedBlocks; }

// One orthogonalisation step on `grid` co-resident blocks of at most emax elements.
static cudaError_t launch_orth(tdmrg_ctx* c, const KrylovWork* k, OrthArgs a, int grid, int emax) {
    const OrthSlots sl = orth_slots(k, grid, a.nk);
    a.partA = sl.partA;
    a.partB = sl.partB[a.j & 1];
    a.partC = sl.partC[a.j & 1];
    a.nextB = sl.partB[(a.j + 1) & 1];
    a.nextC = sl.partC[(a.j + 1) & 1];
    a.emax = emax;
    // shared memory: w and as many of the newest vectors as fit; at least v_{j-1} and v_j, else nothing is staged
    const size_t row = (size_t)std::max(emax, 1) * sizeof(cplx), cap = (size_t)kOrthSmem / k->orth_per_sm;
    const int fit = (int)std::min<size_t>(cap / row, 64) - 1;
    const bool staged = fit >= std::min(a.nv, 2);
    a.rows = staged ? std::min(a.nv, fit) : 0;
    const size_t smem = staged ? (size_t)(1 + a.rows) * row : 0;
    void* params[] = {&a};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(OB);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const void* f = a.seg.nseg > 0 ? (staged ? (const void*)k_lanczos_orth_t<true, true> : (const void*)k_lanczos_orth_t<true, false>)
                                   : (staged ? (const void*)k_lanczos_orth_t<false, true> : (const void*)k_lanczos_orth_t<false, false>);
    c->launches += 1;
    return cudaLaunchKernelExC(&cfg, f, params);
}

// The Lanczos recursion of n_K steps started at phi (Sec. II.A): V, the tridiagonal and the flags in the
// Krylov workspace of (Q, nk).
int lanczos_build(tdmrg_ctx* c, int a, int b, const cplx* phi, int nk, KrylovWork** out) {
    int64_t n = sector_size(c, a, b);
    if (n == 0) return fail(c, TDMRG_ESECTOR, "Lanczos: empty sector");
    Plan* p = nullptr;
    int rc = get_ham_plan(c, a, b, &p);
    if (rc) return rc;
    KrylovWork* k = nullptr;
    rc = ensure_work(c, a, b, nk, n, &k);
    if (rc) return rc;
    *out = k;
    cudaStream_t s = c->stream;
    // blocks own multiples of kOrthAlign elements, at most one block per SM
    const int64_t units = (n + kOrthAlign - 1) / kOrthAlign;
    const int chunk = (int)(kOrthAlign * ((units + k->orth_grid - 1) / k->orth_grid));
    const int grid = (int)((n + chunk - 1) / chunk);
    launch_pdl(k_norm2, NB, NT, 0, s, phi, n, norm_slots(k));
    launch_pdl(k_init_v0, NB, NT, 0, s, phi, n, (const double2*)norm_slots(k), k->V, k->tri, k->flags, nk, orth_slots(k, grid, nk));
    c->launches += 2;
    for (int j = 0; j < nk; ++j) {
        cplx* vj = k->V + (int64_t)j * n;
        rc = run_plan(c, *p, vj, k->w, k->flags, j);
        if (rc) return rc;
        OrthArgs oa{};
        oa.V = k->V; oa.w = k->w; oa.n = n; oa.nv = j + 1; oa.j = j; oa.nk = nk; oa.tol = c->opts.breakdown_tol;
        oa.tri = k->tri; oa.flags = k->flags; oa.status = c->dstatus; oa.chunk = chunk;
        const cudaError_t le = launch_orth(c, k, oa, grid, (int)std::min<int64_t>(chunk, n));
        if (le != cudaSuccess) return cuda_check(c, le, "Lanczos orthogonalisation launch");
    }
    return TDMRG_OK;
}

int evolve(tdmrg_ctx* c, int a, int b, const cplx* phi, int n_v, const double* t_x, int nk, cplx* const* targets) {
    KrylovWork* k = nullptr;
    int rc = lanczos_build(c, a, b, phi, nk, &k);
    if (rc) return rc;
    const int64_t n = k->n;
    cudaStream_t s = c->stream;
    Times tt{};
    for (int x = 0; x < n_v; ++x) tt.t[x] = t_x[x];
    // equally spaced targets from t = 0 (the TST schedule): one time step's Taylor chain, columns in parallel
    std::vector<int> ord(n_v);
    for (int x = 0; x < n_v; ++x) ord[x] = x;
    std::stable_sort(ord.begin(), ord.end(), [&](int p, int q) { return t_x[p] < t_x[q]; });
    const double tmax = t_x[ord[n_v - 1]];
    bool eq = n_v >= 2 && n_v <= 16 && t_x[ord[0]] == 0.0 && t_x[ord[1]] > 0.0;
    const double dt = eq ? t_x[ord[1]] : 0.0;
    for (int m = 2; m < n_v && eq; ++m) eq = std::fabs(t_x[ord[m]] - m * dt) <= 8.0 * 2.220446049250313e-16 * tmax;
    if (eq) {
        StepTimes st{};
        st.dt = dt; st.n_v = n_v; st.xmax = ord[n_v - 1];
        for (int m = 0; m < n_v; ++m) st.order[m] = ord[m];
        launch_pdl(k_tridiag_exp_eq, k->nk, 32, 0, s, k->tri, k->flags, st, k->coef, k->coef + 16 * 32, k->bar + 2);
    } else {
        launch_pdl(k_tridiag_exp, 1, 32, 0, s, k->tri, k->flags, tt, n_v, k->coef);
    }
    // a target at t = 0 is phi itself: copied (before any target that aliases phi is written), not combined
    std::vector<int> rows;
    for (int x = 0; x < n_v; ++x) {
        if (t_x[x] != 0.0) { rows.push_back(x); continue; }
        if (targets[x] != phi) {
            int rc2 = cuda_check(c, cudaMemcpyAsync(targets[x], phi, (size_t)n * sizeof(cplx), cudaMemcpyDeviceToDevice, s),
                                 "evolve copy");
            if (rc2) return rc2;
        }
    }
    TargetPtrs tg{};
    for (int x = 0; x < n_v; ++x) tg.p[x] = targets[x];
    c->launches += 1 + launch_combine(k->V, n, k->flags, k->coef, rows, tg, c->num_sms, s);
    c->last_krylov = k;
    return cuda_check(c, cudaGetLastError(), "evolve launch");
}

// Ground state in sector Q (ground-state targeting, Sec. II.B): `restarts` times, Lanczos with nk steps from
// psi, the lowest eigenvector of T combined in place into psi.
int ground_state(tdmrg_ctx* c, int a, int b, cplx* psi, int nk, int restarts, double* energy) {
    KrylovWork* k = nullptr;
    for (int r = 0; r < restarts; ++r) {
        int rc = lanczos_build(c, a, b, psi, nk, &k);
        if (rc) return rc;
        launch_pdl(k_tridiag_min, 1, kMinThreads, 0, c->stream, k->tri, k->flags, k->coef);
        TargetPtrs tg{};
        tg.p[0] = psi;
        launch_combine(k->V, k->n, k->flags, k->coef, std::vector<int>{0}, tg, c->num_sms, c->stream);
        c->launches += 2;
        rc = cuda_check(c, cudaGetLastError(), "ground-state launch");
        if (rc) return rc;
    }
    c->last_krylov = k;
    double tri[128];
    int rc = cuda_check(c, cudaMemcpyAsync(tri, k->tri, sizeof(tri), cudaMemcpyDeviceToHost, c->stream), "ground state");
    if (!rc) rc = cuda_check(c, cudaStreamSynchronize(c->stream), "ground state");
    if (!rc) rc = check_device_status(c);
    if (!rc && energy) *energy = tri[T_EMIN];
    return rc;
}

// Device tables of the segmented mode: the CTA partition (each segment gets CTAs in proportion to its
// length, at least one) and the per-segment Krylov state, allocated with the Krylov workspace.
static int ensure_segments(tdmrg_ctx* c, KrylovWork* k, int nseg, const int64_t* seg_len, SegTab* tb, double** tri,
                           int** flags, cplx** coef, int* grid) {
    const int G = k->orth_grid;
    if (nseg < 1 || nseg > G) return fail(c, TDMRG_EINVAL, "evolve_segments: more segments than co-resident blocks");
    const bool same = k->nseg == nseg && std::equal(k->seg_len.begin(), k->seg_len.end(), seg_len) &&
                      (int)k->seg_len.size() == nseg;
    const size_t b_tri = (size_t)nseg * kTriStride * sizeof(double), b_fl = (size_t)nseg * kFlagStride * sizeof(int);
    const size_t b_co = (size_t)nseg * kCoefStride * sizeof(cplx), b_cs = (size_t)G * sizeof(int);
    const size_t b_lo = (size_t)G * sizeof(int64_t), b_c0 = (size_t)(nseg + 1) * sizeof(int);
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t bytes = al(b_tri) + al(b_fl) + al(b_co) + al(b_cs) + 2 * al(b_lo) + al(b_c0);
    unsigned char* m = (unsigned char*)k->segmem;
    if (!same) {
        // partition: CTAs in proportion to the lengths, at least one per segment
        int64_t n = 0;
        for (int s = 0; s < nseg; ++s) n += seg_len[s];
        std::vector<int> cnt(nseg, 1);
        int left = G - nseg;
        for (int s = 0; s < nseg && n > 0; ++s) {
            const int extra = (int)((double)left * (double)seg_len[s] / (double)n);
            cnt[s] += extra;
        }
        int used = 0;
        for (int s = 0; s < nseg; ++s) used += cnt[s];
        for (int s = 0; used < G; s = (s + 1) % nseg) { ++cnt[s]; ++used; }
        std::vector<int> cta_seg, c0(nseg + 1, 0);
        std::vector<int64_t> lo, hi;
        int64_t off = 0;
        for (int s = 0; s < nseg; ++s) {
            c0[s] = (int)cta_seg.size();
            const int64_t ch = (seg_len[s] + cnt[s] - 1) / cnt[s];
            for (int b = 0; b < cnt[s]; ++b) {
                cta_seg.push_back(s);
                lo.push_back(off + std::min(seg_len[s], (int64_t)b * ch));
                hi.push_back(off + std::min(seg_len[s], (int64_t)(b + 1) * ch));
            }
            off += seg_len[s];
        }
        c0[nseg] = (int)cta_seg.size();
        k->seg_emax = 1;
        for (size_t b = 0; b < lo.size(); ++b) k->seg_emax = std::max(k->seg_emax, hi[b] - lo[b]);
        if (k->segmem_bytes < bytes) {
            dev_free(c, k->segmem, k->segmem_bytes);
            k->segmem = nullptr;
            k->segmem_bytes = 0;
            int rc = dev_alloc(c, &k->segmem, bytes, "Krylov segments");
            if (rc) return rc;
            k->segmem_bytes = bytes;
        }
        m = (unsigned char*)k->segmem;
        std::vector<unsigned char> h(al(b_cs) + 2 * al(b_lo) + al(b_c0), 0);
        memcpy(h.data(), cta_seg.data(), b_cs);
        memcpy(h.data() + al(b_cs), lo.data(), b_lo);
        memcpy(h.data() + al(b_cs) + al(b_lo), hi.data(), b_lo);
        memcpy(h.data() + al(b_cs) + 2 * al(b_lo), c0.data(), b_c0);
        int rc = cuda_check(c, cudaMemcpyAsync(m + al(b_tri) + al(b_fl) + al(b_co), h.data(), h.size(), cudaMemcpyHostToDevice,
                                               c->stream), "Krylov segments");
        if (!rc) rc = cuda_check(c, cudaMemsetAsync(m, 0, al(b_tri) + al(b_fl) + al(b_co), c->stream), "Krylov segments");
        if (!rc) rc = cuda_check(c, cudaStreamSynchronize(c->stream), "Krylov segments");
        if (rc) return rc;
        k->nseg = nseg;
        k->seg_len.assign(seg_len, seg_len + nseg);
    }
    *tri = (double*)m;
    *flags = (int*)(m + al(b_tri));
    *coef = (cplx*)(m + al(b_tri) + al(b_fl));
    unsigned char* t = m + al(b_tri) + al(b_fl) + al(b_co);
    tb->cta_seg = (const int*)t;
    tb->cta_lo = (const int64_t*)(t + al(b_cs));
    tb->cta_hi = (const int64_t*)(t + al(b_cs) + al(b_lo));
    tb->seg_cta0 = (const int*)(t + al(b_cs) + 2 * al(b_lo));
    tb->nseg = nseg;
    *grid = G;
    return TDMRG_OK;
}

// Independent Krylov advances side by side (Sec. II.A, Eq. lanczosevolution for each segment): one H psi
// over the whole vector per Lanczos step (the superblock is a direct sum, so its products never mix
// segments), orthogonalisation, tridiagonal exponentials and targets per segment.
int evolve_segments(tdmrg_ctx* c, int a, int b, const cplx* phi, int nseg, const int64_t* seg_len, int n_v,
                    const double* t_x, int nk, cplx* const* targets) {
    const int64_t n = sector_size(c, a, b);
    if (n == 0) return fail(c, TDMRG_ESECTOR, "evolve_segments: empty sector");
    int64_t tot = 0;
    for (int s = 0; s < nseg; ++s) {
        if (seg_len[s] < 1) return fail(c, TDMRG_EINVAL, "evolve_segments: empty segment");
        tot += seg_len[s];
    }
    if (tot != n) return fail(c, TDMRG_EINVAL, "evolve_segments: the segment lengths do not add up to the sector size");
    Plan* p = nullptr;
    int rc = get_ham_plan(c, a, b, &p);
    if (rc) return rc;
    KrylovWork* k = nullptr;
    rc = ensure_work(c, a, b, nk, n, &k);
    if (rc) return rc;
    SegTab tb{};
    double* tri = nullptr;
    int* flags = nullptr;
    cplx* coef = nullptr;
    int G = 0;
    rc = ensure_segments(c, k, nseg, seg_len, &tb, &tri, &flags, &coef, &G);
    if (rc) return rc;
    cudaStream_t s = c->stream;
    launch_pdl(k_norm2_seg, G, NT, 0, s, phi, tb, norm_slots(k));
    launch_pdl(k_init_v0_seg, G, NT, 0, s, phi, tb, (const double2*)norm_slots(k), k->V, tri, flags, nk, orth_slots(k, G, nk));
    c->launches += 2;
    for (int j = 0; j < nk; ++j) {
        cplx* vj = k->V + (int64_t)j * n;
        rc = run_plan(c, *p, vj, k->w, nullptr, 0);   // every segment's product (a stopped one's is ignored)
        if (rc) return rc;
        OrthArgs oa{};
        oa.V = k->V; oa.w = k->w; oa.n = n; oa.nv = j + 1; oa.j = j; oa.nk = nk; oa.tol = c->opts.breakdown_tol;
        oa.tri = tri; oa.flags = flags; oa.status = c->dstatus; oa.seg = tb;
        const cudaError_t le = launch_orth(c, k, oa, G, (int)k->seg_emax);
        if (le != cudaSuccess) return cuda_check(c, le, "segmented Lanczos launch");
    }
    Times tt{};
    for (int x = 0; x < n_v; ++x) tt.t[x] = t_x[x];
    launch_pdl(k_tridiag_exp, nseg, 32, 0, s, tri, flags, tt, n_v, coef);
    TargetPtrs tg{};
    for (int x = 0; x < n_v; ++x) tg.p[x] = targets[x];
    std::vector<int> rows(n_v);
    for (int x = 0; x < n_v; ++x) rows[x] = x;
    const CombineList cl = combine_list(rows, tg);
    launch_pdl(k_combine_seg, dim3(G, cl.n), CBT, 0, s, k->V, n, tb, flags, coef, cl);
    c->launches += 2;
    return cuda_check(c, cudaGetLastError(), "evolve_segments launch");
}

// Krylov dimension used and error estimate of each segment of the last evolve_segments on (Q, nk).
int segments_info(tdmrg_ctx* c, int a, int b, int nk, int nseg, int* nk_used, double* err) {
    auto it = c->krylov.find(std::make_pair(a * 4096 + b, nk));
    if (it == c->krylov.end() || it->second.nseg != nseg || !it->second.segmem)
        return fail(c, TDMRG_ESTATE, "evolve_segments_info: no segmented evolve with these arguments");
    std::vector<double> tri((size_t)nseg * kTriStride);
    std::vector<int> fl((size_t)nseg * kFlagStride);
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const unsigned char* m = (const unsigned char*)it->second.segmem;
    int rc = cuda_check(c, cudaMemcpyAsync(tri.data(), m, tri.size() * sizeof(double), cudaMemcpyDeviceToHost, c->stream), "info");
    if (!rc) rc = cuda_check(c, cudaMemcpyAsync(fl.data(), m + al(tri.size() * sizeof(double)), fl.size() * sizeof(int),
                                                cudaMemcpyDeviceToHost, c->stream), "info");
    if (!rc) rc = cuda_check(c, cudaStreamSynchronize(c->stream), "info");
    if (!rc) rc = check_device_status(c);
    if (rc) return rc;
    for (int s = 0; s < nseg; ++s) {
        if (nk_used) nk_used[s] = fl[(size_t)s * kFlagStride];
        if (err) err[s] = tri[(size_t)s * kTriStride + T_ERR];
    }
    return TDMRG_OK;
}

int evolve_info(tdmrg_ctx* c, int* nk_used, double* err, double* alpha, double* beta) {
    KrylovWork* k = c->last_krylov;
    double tri[128];
    int flags[4];
    int rc = cuda_check(c, cudaMemcpyAsync(tri, k->tri, sizeof(tri), cudaMemcpyDeviceToHost, c->stream), "evolve_info");
    if (!rc) rc = cuda_check(c, cudaMemcpyAsync(flags, k->flags, sizeof(flags), cudaMemcpyDeviceToHost, c->stream), "evolve_info");
    if (!rc) rc = cuda_check(c, cudaStreamSynchronize(c->stream), "evolve_info sync");
    if (rc) return rc;
    rc = check_device_status(c);
    if (rc) return rc;
    if (nk_used) *nk_used = flags[0];
    if (err) *err = tri[T_ERR];
    for (int j = 0; j < flags[0]; ++j) {
        if (alpha) alpha[j] = tri[T_ALPHA + j];
        if (beta) beta[j] = tri[T_BETA + j];
    }
    return TDMRG_OK;
}

}  // namespace tdmrg
