// Numbers held as the unevaluated sum of two FP32 values (about 47 bits), for
// plan-time transforms whose results are rounded to FP32: FP64 instructions
// run at 1/64 of the FP32 rate on this GPU, a sum of pairs costs 11 FP32
// operations and a product 7 (T. J. Dekker, Numer. Math. 18 (1971) 224-242;
// D. E. Knuth, TAOCP 2, 4.2.2).  The range is FP32's, so the values must be
// scaled to order 1.
//
// Spectra rounded to FP32 from pairs serve as well as from FP64: the forward of an
// FP32 plan differs from the FP64 plan's by the same 1.4e-7 to 2.9e-7 a component,
// to three digits, with either (17 x 9 x 40 and 20 x 700 x 12 cells, the second
// with stations 100 cell edges up; nine components, means of four densities).
#pragma once
#include "fft_block.cuh"

namespace grav {

struct alignas(8) pairf {
    float h, l;
    pairf() = default;
    __host__ __device__ constexpr pairf(float hi, float lo) : h(hi), l(lo) {}
    __host__ __device__ constexpr pairf(double v) : h((float)v), l((float)(v - (double)(float)v)) {}
};
struct alignas(16) pairf2 { pairf x, y; };
template <> struct cplx<pairf> { using type = pairf2; };

// a + b with |a| >= |b|: sum and its rounding error.
__device__ __forceinline__ pairf quick_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return pairf(s, __fsub_rn(b, __fsub_rn(s, a)));
}
// a + b: sum and its rounding error.
__device__ __forceinline__ pairf two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
    return pairf(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z)));
}
__device__ __forceinline__ pairf operator-(pairf a) { return pairf(-a.h, -a.l); }
__device__ __forceinline__ pairf operator+(pairf a, pairf b) {
    const pairf s = two_sum(a.h, b.h);
    return quick_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ pairf operator-(pairf a, pairf b) { return a + (-b); }
__device__ __forceinline__ pairf operator*(pairf a, pairf b) {
    const float p = __fmul_rn(a.h, b.h);
    const float e = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)));
    return quick_sum(p, e);
}
// a b + c d with one normalisation.
__device__ __forceinline__ pairf dot2(pairf a, pairf b, pairf c, pairf d) {
    const float p = __fmul_rn(a.h, b.h), q = __fmul_rn(c.h, d.h);
    const float pe = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.h, -p)));
    const float qe = __fmaf_rn(c.h, d.l, __fmaf_rn(c.l, d.h, __fmaf_rn(c.h, d.h, -q)));
    const pairf s = two_sum(p, q);
    return quick_sum(s.h, __fadd_rn(s.l, __fadd_rn(pe, qe)));
}
template <> __device__ __forceinline__ pairf2 cmul<pairf2>(pairf2 a, pairf2 b) {
    return cmk<pairf2>(dot2(a.x, b.x, -a.y, b.y), dot2(a.x, b.y, a.y, b.x));
}

}  // namespace grav
