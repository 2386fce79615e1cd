// Float-float ("paired FP32") scalar arithmetic: a value is h + l, two FP32
// words with |l| <= ulp(h) / 2, about 48 significant bits.  The sums and
// products are Dekker's (T. J. Dekker, "A floating-point technique for
// extending the available precision", Numer. Math. 18, 1971): TwoSum
// (Knuth) for the head words, the product's rounding error by FMA, the low
// words added in FP32.  Reciprocal and reciprocal square root take the FP32
// result and one correction from its residual in pairs.
// On GB300 an FP64 warp instruction occupies the SM sub-partition's FP64
// pipe for 64 cycles whether one lane or 32 are active; these run on the
// FP32 pipe (4-cycle latency, full rate) and serve the per-column scalars
// of the paired-FP32 kernels.
#pragma once

namespace tlr {

struct FF {
    float h, l;
};

__device__ __forceinline__ FF ff_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return FF{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ FF ff_fast(float a, float b) {  // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const FF s = ff_two_sum(a.h, b.h);
    return ff_fast(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ FF ff_neg(FF a) { return FF{-a.h, -a.l}; }
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return ff_fast(p, e);
}
// 1 / sqrt(a), a > 0: the FP32 approximation y and its residual e = 1 - a y^2
// in pairs, then y + y (e / 2 + 3 e^2 / 8) (the third-order step; e ~ 2^-22).
// One chain of FP32 operations, where a square root and a quotient take two
// IEEE square roots and divisions one after the other.
__device__ __forceinline__ FF ff_rsqrt(FF a) {
    const float y = rsqrtf(a.h);
    const FF ay = ff_mul(a, FF{y, 0.f});
    const float p = __fmul_rn(ay.h, y), pe = __fmaf_rn(ay.l, y, __fmaf_rn(ay.h, y, -p));
    const float e = __fsub_rn(__fsub_rn(1.0f, p), pe);
    return ff_fast(y, __fmul_rn(y, __fmul_rn(e, __fmaf_rn(0.375f, e, 0.5f))));
}
// 1 / a, a != 0 and normal: the FP32 reciprocal y, then y + y (e + e^2), e = 1 - a y
__device__ __forceinline__ FF ff_rcp(FF a) {
    const float y = __frcp_rn(a.h);
    const float p = __fmul_rn(a.h, y), pe = __fmaf_rn(a.l, y, __fmaf_rn(a.h, y, -p));
    const float e = __fsub_rn(__fsub_rn(1.0f, p), pe);
    return ff_fast(y, __fmul_rn(y, __fmaf_rn(e, e, e)));
}

}  // namespace tlr
