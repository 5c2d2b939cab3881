// Double-float arithmetic: a real number held as the unevaluated sum hi + lo
// of two floats (|lo| <= ulp(hi) / 2), about 48 significant bits, computed
// on the FP32 units.  The sum takes Knuth's two-sum of the high parts, adds
// the low parts into its error term and renormalises with a second two-sum
// (after cancellation the high sum can be smaller than that term, which a
// fast two-sum would get wrong): its error is about 2^-48 times |a| + |b|,
// what a transform's norm-wise error analysis needs.  The product forms the
// exact product of the high parts with a fused multiply-add, adds the cross
// terms and renormalises with a fast two-sum (the high product dominates).
//
// The kernels work on complex numbers (cdf, below), whose real and imaginary
// parts go through these steps together on the paired FP32 instructions: half
// the instructions of the scalar form, whose unrolled transforms waited on
// instruction fetch.  The double-float product at 256^3 took 33.0 ms with
// scalar operations and conversion instructions at both ends, 20 ms this way,
// with the same error against 64 bits (2.96e-15 relative, the mean over 34
// lattices).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace dda {

struct DF {
    float hi, lo;
    DF() = default;
    // the double rounded to the nearest float, plus the rounded remainder
    __host__ __device__ __forceinline__ DF(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
    __host__ __device__ __forceinline__ DF(float h, float l) : hi(h), lo(l) {}
};

// Scalar operations: the reference form of the steps, checked on the host
// against exact arithmetic; the kernels run their paired forms below.
//
// The high product, rounded on its own: the device compiler never contracts
// __fmul_rn into the sum that follows it, which would count the product's
// rounding error twice.
__host__ __device__ __forceinline__ float df_mul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}

__host__ __device__ __forceinline__ DF df_fast_two_sum(float a, float b) {   // |a| >= |b|
    const float s = a + b;
    return DF(s, b - (s - a));
}
__host__ __device__ __forceinline__ DF df_two_sum(float a, float b) {   // any magnitudes
    const float s = a + b;
    const float v = s - a;
    return DF(s, (a - (s - v)) + (b - v));
}
__host__ __device__ __forceinline__ DF operator+(DF a, DF b) {
    const DF s = df_two_sum(a.hi, b.hi);
    return df_two_sum(s.hi, s.lo + (a.lo + b.lo));
}
__host__ __device__ __forceinline__ DF operator-(DF a) { return DF(-a.hi, -a.lo); }
__host__ __device__ __forceinline__ DF operator-(DF a, DF b) { return a + (-b); }
__host__ __device__ __forceinline__ DF operator*(DF a, DF b) {
    const float p = df_mul(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);   // the exact error of the high product
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df_fast_two_sum(p, e);
}
// a * b + c (with float and double overloads, so that the name does not
// hide the math library's inside this namespace)
__host__ __device__ __forceinline__ DF fma(DF a, DF b, DF c) { return a * b + c; }
__host__ __device__ __forceinline__ float fma(float a, float b, float c) { return ::fmaf(a, b, c); }
__host__ __device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }

// Complex double-float, 16 bytes: the high parts of (re, im), then the low
// parts.  On the device both parts go through the arithmetic as one pair, on
// the paired FP32 instructions (add.f32x2 and its kin), so that a complex
// operation takes the instructions of a real one.
struct __align__(16) cdf {
    float2 h, l;
};
__host__ __device__ __forceinline__ cdf make_cdf(DF re, DF im) {
    return cdf{make_float2(re.hi, im.hi), make_float2(re.lo, im.lo)};
}

#ifdef __CUDACC__
// Conversions between double and double-float on the integer units (a
// conversion instruction between the two widths, like any FP64 one, takes 16
// cycles of an SM per warp): hi is the double rounded to 24 bits, lo the
// signed 29-bit rest.  Doubles outside 2^-70 .. 2^126, zeros among them, and
// floats that are not normal numbers take the conversion instructions.
__device__ __forceinline__ DF df_split(double d) {
    const uint64_t b = (uint64_t)__double_as_longlong(d);
    const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu, sign = (uint32_t)(b >> 63) << 31;
    if (e - 953u > 1149u - 953u) return DF(d);
    const uint32_t hi = (uint32_t)((((b & 0x7fffffffffffffffull) + (1u << 28)) >> 29) - (896ull << 23));
    const int rest = ((int)((uint32_t)b << 3)) >> 3;
    return DF(__uint_as_float(hi | sign), (float)rest * __uint_as_float(((e - 948u) << 23) | sign));
}
__device__ __forceinline__ double df_widen(float f) {
    const uint32_t b = __float_as_uint(f), e = (b >> 23) & 0xffu;
    if (e - 1u > 253u) return (double)f;
    return __longlong_as_double((long long)(((uint64_t)(b >> 31) << 63) | ((uint64_t)(b & 0x7fffffffu) << 29)) +
                                (896ll << 52));
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    float2 d;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long&>(d))
        : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
    return d;
}
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }

// s + t renormalised, |t| a few ulps of the terms that made s.  A fast
// two-sum: where cancellation has left |s| < |t| it drops at most an ulp of
// t, 2^-48 of those terms.  (Over 256-point transforms the error is the
// same to all digits as with a full two-sum, which costs three operations
// more.)
__device__ __forceinline__ cdf df_renorm(float2 s, float2 t) {
    const float2 r = add2(s, t);
    return cdf{r, sub2(t, sub2(r, s))};
}
__device__ __forceinline__ cdf df_add(cdf a, cdf b) {
    const float2 s = add2(a.h, b.h), v = sub2(s, a.h);
    const float2 e = add2(sub2(a.h, sub2(s, v)), sub2(b.h, v));
    return df_renorm(s, add2(e, add2(a.l, b.l)));
}
__device__ __forceinline__ cdf df_sub(cdf a, cdf b) {
    const float2 s = sub2(a.h, b.h), v = sub2(s, a.h);
    const float2 e = sub2(sub2(a.h, sub2(s, v)), add2(b.h, v));
    return df_renorm(s, add2(e, sub2(a.l, b.l)));
}
// elementwise products a b of the two lanes.  The high product is formed
// negated, so that its exact error comes from one fused multiply-add.
// (Sums of products that skip the renormalisation of each, as in a
// compensated dot product, save a quarter of a complex product's operations
// but raise the transforms' error by 9%.)
__device__ __forceinline__ cdf df_mul2(float2 ah, float2 al, float2 bh, float2 bl) {
    const float2 p = __fmul2_rn(make_float2(-ah.x, -ah.y), bh);
    float2 e = __ffma2_rn(ah, bh, p);
    e = __ffma2_rn(ah, bl, e);
    e = __ffma2_rn(al, bh, e);
    const float2 r = sub2(e, p);
    return cdf{r, sub2(e, add2(r, p))};
}
// complex product: a.x (b.x, b.y) + a.y (-b.y, b.x)
__device__ __forceinline__ float2 turned(float2 b) { return make_float2(-b.y, b.x); }
__device__ __forceinline__ cdf df_cmul(cdf a, cdf b) {
    return df_add(df_mul2(both(a.h.x), both(a.l.x), b.h, b.l),
                  df_mul2(both(a.h.y), both(a.l.y), turned(b.h), turned(b.l)));
}
// acc + a b, one product at a time (adding the complex product whole raised
// the matrix product's error by 5%)
__device__ __forceinline__ cdf df_cfma(cdf a, cdf b, cdf acc) {
    return df_add(df_add(acc, df_mul2(both(a.h.y), both(a.l.y), turned(b.h), turned(b.l))),
                  df_mul2(both(a.h.x), both(a.l.x), b.h, b.l));
}
__device__ __forceinline__ cdf df_cscale(cdf a, DF s) { return df_mul2(both(s.hi), both(s.lo), a.h, a.l); }
#endif

}  // namespace dda
