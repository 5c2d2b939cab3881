// Double-float ("hi + lo") arithmetic: a number held as the unevaluated sum
// of two floats (|lo| <= ulp(hi) / 2), about 48 significant bits, computed
// on the FP32 units.  The kernels work on complex numbers (cdf, below), whose
// real and imaginary parts go through every step together on the paired FP32
// instructions: half the instructions of a scalar form, whose unrolled
// transforms waited on instruction fetch (product at 256^3: 33 ms with scalar
// operations and conversion instructions at both ends, 19.2 ms this way, with
// the same error against 64 bits: 2.96e-15 relative, the mean over 34 lattices).
//
// The sum takes Knuth's two-sum of the high parts, adds the low parts into
// its error term and renormalises with a fast two-sum: its error is at most
// 3 2^-48 of |a| + |b|, what a transform's norm-wise error analysis needs.  The
// fast two-sum is exact although after cancellation the high sum s can be
// smaller than the term t added to it: s is then a multiple of the last place
// of the smaller operand, and so of t's, which is all that it needs.  The
// product forms the exact product of the high parts with a fused
// multiply-add, adds the cross terms and renormalises in the same way.
//
// Everything here compiles for the host too, with plain float operations
// (which a host compiler must not contract) in place of the paired
// instructions, and is checked there against exact arithmetic.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace dda {

struct DF {
    float hi, lo;
    DF() = default;
    // the double rounded to the nearest float, plus the rounded remainder
    __host__ __device__ __forceinline__ DF(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
    __host__ __device__ __forceinline__ DF(float h, float l) : hi(h), lo(l) {}
};

// fused multiply-add of either width
__host__ __device__ __forceinline__ float fma(float a, float b, float c) { return ::fmaf(a, b, c); }
__host__ __device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }

// Complex double-float, 16 bytes: the high parts of (re, im), then the low
// parts.
struct __align__(16) cdf {
    float2 h, l;
};
__host__ __device__ __forceinline__ cdf make_cdf(DF re, DF im) {
    return cdf{make_float2(re.hi, im.hi), make_float2(re.lo, im.lo)};
}

// bit patterns
template <typename To, typename From> __host__ __device__ __forceinline__ To bits_as(From v) {
    static_assert(sizeof(To) == sizeof(From), "same width");
    To r;
    memcpy(&r, &v, sizeof r);
    return r;
}

// Conversions between double and double-float on the integer units (a
// conversion instruction between the two widths, like any FP64 one, takes 16
// cycles of an SM per warp): hi is the double rounded to 24 bits (a tie away
// from zero, lo is then half an ulp the other way), lo the signed 29-bit rest.
// Doubles outside 2^-70 .. 2^126, zeros among them, and floats that are not
// normal numbers take the conversion instructions.
__host__ __device__ __forceinline__ DF df_split(double d) {
    const uint64_t b = bits_as<uint64_t>(d);
    const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu, sign = (uint32_t)(b >> 63) << 31;
    if (e - 953u > 1149u - 953u) return DF(d);
    const uint32_t hi = (uint32_t)((((b & 0x7fffffffffffffffull) + (1u << 28)) >> 29) - (896ull << 23));
    const int rest = ((int)((uint32_t)b << 3)) >> 3;
    return DF(bits_as<float>(hi | sign), (float)rest * bits_as<float>(((e - 948u) << 23) | sign));
}
__host__ __device__ __forceinline__ double df_widen(float f) {
    const uint32_t b = bits_as<uint32_t>(f), e = (b >> 23) & 0xffu;
    if (e - 1u > 253u) return (double)f;
    return bits_as<double>((uint64_t)(((uint64_t)(b >> 31) << 63) | ((uint64_t)(b & 0x7fffffffu) << 29)) + (896ull << 52));
}

// paired operations, each rounded on its own
__host__ __device__ __forceinline__ float2 add2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    return __fadd2_rn(a, b);
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__host__ __device__ __forceinline__ float2 sub2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    float2 d;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long&>(d))
        : "l"(reinterpret_cast<unsigned long long&>(a)), "l"(reinterpret_cast<unsigned long long&>(b)));
    return d;
#else
    return make_float2(a.x - b.x, a.y - b.y);
#endif
}
__host__ __device__ __forceinline__ float2 mul2(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    return __fmul2_rn(a, b);
#else
    return make_float2(a.x * b.x, a.y * b.y);
#endif
}
__host__ __device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
#ifdef __CUDA_ARCH__
    return __ffma2_rn(a, b, c);
#else
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
__host__ __device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }

// s + t renormalised (a fast two-sum, see above; a full one takes three
// operations more and gives 256-point transforms the same error to all digits)
__host__ __device__ __forceinline__ cdf df_renorm(float2 s, float2 t) {
    const float2 r = add2(s, t);
    return cdf{r, sub2(t, sub2(r, s))};
}
__host__ __device__ __forceinline__ cdf df_add(cdf a, cdf b) {
    const float2 s = add2(a.h, b.h), v = sub2(s, a.h);
    const float2 e = add2(sub2(a.h, sub2(s, v)), sub2(b.h, v));
    return df_renorm(s, add2(e, add2(a.l, b.l)));
}
__host__ __device__ __forceinline__ cdf df_sub(cdf a, cdf b) {
    const float2 s = sub2(a.h, b.h), v = sub2(s, a.h);
    const float2 e = sub2(sub2(a.h, sub2(s, v)), add2(b.h, v));
    return df_renorm(s, add2(e, sub2(a.l, b.l)));
}
// elementwise products a b of the two lanes.  The high product is formed
// negated, so that its exact error comes from one fused multiply-add.
// (Sums of products that skip the renormalisation of each, as in a
// compensated dot product, save a quarter of a complex product's operations
// and 10% of the 128^3 matrix product's time, but raise the error of 256-point
// transforms by 9% and the matrix product's by 13%.)
__host__ __device__ __forceinline__ cdf df_mul2(float2 ah, float2 al, float2 bh, float2 bl) {
    const float2 p = mul2(make_float2(-ah.x, -ah.y), bh);
    float2 e = fma2(ah, bh, p);
    e = fma2(ah, bl, e);
    e = fma2(al, bh, e);
    const float2 r = sub2(e, p);
    return cdf{r, sub2(e, add2(r, p))};
}
// complex product: a.x (b.x, b.y) + a.y (-b.y, b.x)
__host__ __device__ __forceinline__ float2 turned(float2 b) { return make_float2(-b.y, b.x); }
__host__ __device__ __forceinline__ cdf df_cmul(cdf a, cdf b) {
    return df_add(df_mul2(both(a.h.x), both(a.l.x), b.h, b.l),
                  df_mul2(both(a.h.y), both(a.l.y), turned(b.h), turned(b.l)));
}
// acc + a b, one product at a time (adding the complex product whole raised
// the matrix product's error by 5%)
__host__ __device__ __forceinline__ cdf df_cfma(cdf a, cdf b, cdf acc) {
    return df_add(df_add(acc, df_mul2(both(a.h.y), both(a.l.y), turned(b.h), turned(b.l))),
                  df_mul2(both(a.h.x), both(a.l.x), b.h, b.l));
}
__host__ __device__ __forceinline__ cdf df_cscale(cdf a, DF s) { return df_mul2(both(s.hi), both(s.lo), a.h, a.l); }

}  // namespace dda
