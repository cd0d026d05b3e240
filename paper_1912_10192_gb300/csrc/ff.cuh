// ff.cuh -- numbers carried as an unevaluated sum of two binary32 values
// ("double-float", Dekker 1971; the operations after Knuth's two-sum and the
// fused-multiply-add product), about 46 bits, on the FP32 pipe.
//
// The FP64 pipe retires two lanes per SM and cycle, the FP32 pipe 128: an FP64
// warp instruction holds its scheduler's share of the FP64 pipe for 64 cycles,
// a product below takes 5 issue slots and a sum 11, while that pipe stays free
// for other work. These numbers stand in where 46 bits change no result: in
// iterations whose last step is taken from FP64 residuals.
//
// Range: that of binary32. Callers scale by powers of two (exact) so that
// values are O(1); a value below 2^-74 keeps one word, one below 2^-126 is 0.
#pragma once
#include <cuda_runtime.h>

#include "cvt.cuh"

namespace hamr {

struct ff {
    float h, l;
};

// x 2^(sh >> 20) with the 24 leading fraction bits of x in h and the other 29, rounded to 24, in l,
// from the bit patterns (no FP64 instruction); sh: a multiple of 2^20. Infinities, NaNs and values
// above binary32's range give non-finite or meaningless words: callers test the result they need.
__device__ __forceinline__ ff ff_of(double x, int sh = 0) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int a = (int)((hi & 0x7fffffffu) + (unsigned)sh);  // wraps: sh may be several exponents' sum
    const unsigned s = hi & 0x80000000u;
    const unsigned u = (((unsigned)a - 0x38000000u) << 3) | (lo >> 29);  // binary32 bits of the truncated value
    const float r = (float)(lo & 0x1fffffffu);
    // the dropped bits count 2^(e - 52): exponent field of h minus 52
    float l = r * __uint_as_float((u & 0x7f800000u) - (52u << 23));
    ff o;
    o.h = __uint_as_float(a < 0x38100000 ? 0u : (u | s));
    l = a < 0x3b500000 ? 0.0f : l;
    o.l = __uint_as_float(__float_as_uint(l) ^ s);
    return o;
}

__device__ __forceinline__ double ff_d(ff a) { return widen(a.h) + widen(a.l); }

__device__ __forceinline__ ff ff_neg(ff a) { return ff{-a.h, -a.l}; }
__device__ __forceinline__ ff ff_scale(ff a, float p) { return ff{a.h * p, a.l * p}; }  // p a power of two

// product: the rounding error of the leading product by one fused multiply-add, the cross products
// and the product of the low words added to it (relative error of a few 2^-47)
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.l, b.l, e);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return ff{p, e};
}

// sum: two-sum of the leading words, the low words added to its error, renormalised
__device__ __forceinline__ ff ff_add(ff a, ff b) {
    const float s = __fadd_rn(a.h, b.h);
    const float t = __fsub_rn(s, a.h);
    float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    e = __fadd_rn(e, __fadd_rn(a.l, b.l));
    const float h = __fadd_rn(s, e);
    return ff{h, __fsub_rn(e, __fsub_rn(h, s))};
}
__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }
__device__ __forceinline__ ff ff_norm(ff a) {
    const float h = __fadd_rn(a.h, a.l);
    return ff{h, __fsub_rn(a.l, __fsub_rn(h, a.h))};
}

// the hardware's approximate reciprocal (2^-23)
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 1 / x: the approximate reciprocal and one Newton correction in the low word
__device__ __forceinline__ ff ff_rcp(ff x) {
    const float r = rcp_approx(x.h);
    float e = __fmaf_rn(-x.h, r, 1.0f);
    e = __fmaf_rn(-x.l, r, e);
    return ff{r, r * e};
}

// 1 / sqrt(x), x > 0: y = approximate reciprocal square root, e = 1 - x y^2, y (1 + e/2 + 3 e^2/8)
__device__ __forceinline__ ff ff_rsqrt(ff x) {
    const float y = rsqrtf(x.h);
    const float p = __fmul_rn(y, y), q = __fmaf_rn(y, y, -p);
    float e = __fmaf_rn(-x.h, p, 1.0f);
    e = __fmaf_rn(-x.h, q, e);
    e = __fmaf_rn(-x.l, p, e);
    return ff{y, y * (e * __fmaf_rn(0.375f, e, 0.5f))};
}

// sqrt(x), 0 for x <= 0: s = x / sqrt(x) in binary32, corrected by (x - s^2) / (2 sqrt(x))
__device__ __forceinline__ ff ff_sqrt_pos(ff x) {
    if (!(x.h > 0.0f)) return ff{0.0f, 0.0f};
    const float y = rsqrtf(x.h);
    const float s = __fmul_rn(x.h, y);
    const float r = __fadd_rn(__fmaf_rn(-s, s, x.h), x.l);
    return ff{s, r * (0.5f * y)};
}

__device__ __forceinline__ bool ff_less(ff a, ff b) {  // of normalised numbers
    return a.h < b.h || (a.h == b.h && a.l < b.l);
}

}  // namespace hamr
