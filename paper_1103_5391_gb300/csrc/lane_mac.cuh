// Multiply-adds of one output per lane in FP64, shared by the grouped GEMM (gemm_f64.cu) and the thin products of the
// tensor kernel (ozaki.cu): operands straight from global memory, UK k-steps ahead of their use (4 in the grouped GEMM;
// 2 in the thin products, which share the register file with the tensor pipeline's epilogue: 4 spill there).
#pragma once

namespace tdmrg {

// s0 += Re a Re b, s1 += Im a Im b, s2 += Re a Im b, s3 += Im a Re b over k in [k0, k1)
template <int MODE, int UK>
__device__ __forceinline__ void seg_mac(const double2* __restrict__ pa, const double2* __restrict__ pb, int ak, int bk, int nk,
                                        double (&s)[4]) {
    auto mac = [&](double2 a, double2 b) {
        s[0] = fma(a.x, b.x, s[0]);
        if (MODE == 0) s[1] = fma(a.y, b.y, s[1]);
        if (MODE != 2) s[2] = fma(a.x, b.y, s[2]);
        if (MODE != 1) s[3] = fma(a.y, b.x, s[3]);
    };
    int k = 0;
    if (nk >= UK) {
        double2 a[UK], b[UK];
#pragma unroll
        for (int u = 0; u < UK; ++u) { a[u] = __ldg(pa + u * ak); b[u] = __ldg(pb + u * bk); }
        for (k = UK; k + UK <= nk; k += UK) {
            pa += (int64_t)UK * ak;
            pb += (int64_t)UK * bk;
            double2 na[UK], nb[UK];
#pragma unroll
            for (int u = 0; u < UK; ++u) { na[u] = __ldg(pa + u * ak); nb[u] = __ldg(pb + u * bk); }
#pragma unroll
            for (int u = 0; u < UK; ++u) mac(a[u], b[u]);
#pragma unroll
            for (int u = 0; u < UK; ++u) { a[u] = na[u]; b[u] = nb[u]; }
        }
        pa += (int64_t)UK * ak;
        pb += (int64_t)UK * bk;
#pragma unroll
        for (int u = 0; u < UK; ++u) mac(a[u], b[u]);
    }
    for (; k < nk; ++k) {
        mac(__ldg(pa), __ldg(pb));
        pa += ak;
        pb += bk;
    }
}

}  // namespace tdmrg
