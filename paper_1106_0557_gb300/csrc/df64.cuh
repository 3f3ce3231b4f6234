// df64.cuh -- float-float ("double-single") arithmetic for an FP64-class
// solve on the FP32 units.
//
// A value is hi + lo with |lo| <= ulp(hi) / 2, about 48 significant bits.
// The building blocks are the error-free transformations of Knuth (two-sum)
// and Dekker (fast two-sum), and the fused multiply-add for the exact
// product error:
//   add: (s, e) = two_sum(a.hi, b.hi); e += a.lo + b.lo; fast_two_sum(s, e)
//        -- the "sloppy" sum, whose error is relative to |a| + |b|, which is
//        the bound an FFT's normwise error analysis uses anyway;
//   mul: p = a.hi b.hi; e = fma(a.hi, b.hi, -p) + a.hi b.lo + a.lo b.hi;
//        fast_two_sum(p, e).
// Only sums and explicit fma() calls appear, so contraction of a * b + c by
// the compiler cannot change the rounding of the error-free steps.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace isofft {

struct df64 {
    float hi, lo;
    df64() = default;
    __host__ __device__ constexpr df64(float h, float l) : hi(h), lo(l) {}
    // exact split of a double into the nearest float and the float nearest
    // to the remainder
    __host__ __device__ constexpr df64(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
    __host__ __device__ constexpr explicit df64(int i) : hi((float)i), lo(0.0f) {}
    __host__ __device__ constexpr double to_double() const { return (double)hi + (double)lo; }
};

__host__ __device__ __forceinline__ df64 df64_fast_two_sum(float a, float b)
{
    const float s = a + b;
    return {s, b - (s - a)};
}

__host__ __device__ __forceinline__ df64 operator+(df64 a, df64 b)
{
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    float e = (a.hi - (s - bb)) + (b.hi - bb);
    e += a.lo + b.lo;
    return df64_fast_two_sum(s, e);
}

// The sum without its closing renormalisation: hi = fl(a.hi + b.hi) and lo
// its exact error plus a.lo + b.lo.  hi + lo is the same sloppy sum, but lo
// may exceed half an ulp of hi (by a few ulps along a chain of such sums,
// and more where hi cancels).  The FFT engine's butterflies chain these and
// renormalise (df64_renorm) before any product, whose error term drops
// lo x lo and so needs |lo| << |hi|.
__host__ __device__ __forceinline__ df64 df64_add_lazy(df64 a, df64 b)
{
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    const float e = (a.hi - (s - bb)) + (b.hi - bb);
    return {s, e + (a.lo + b.lo)};
}
// The product without its closing renormalisation (its lo is the exact
// error of hi plus the cross terms, within a few ulps of hi): for products
// that only enter sums.  Both operands must be normalised.
__host__ __device__ __forceinline__ df64 df64_mul_lazy(df64 a, df64 b)
{
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return {p, e};
}
__host__ __device__ __forceinline__ df64 df64_renorm(df64 a)
{
    return df64_fast_two_sum(a.hi, a.lo);
}

__host__ __device__ __forceinline__ df64 operator-(df64 a) { return {-a.hi, -a.lo}; }
__host__ __device__ __forceinline__ df64 operator-(df64 a, df64 b) { return a + (-b); }

__host__ __device__ __forceinline__ df64 operator*(df64 a, df64 b)
{
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df64_fast_two_sum(p, e);
}

__host__ __device__ __forceinline__ bool operator>(df64 a, df64 b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }

// Bit patterns, on the device and on the host.
__host__ __device__ __forceinline__ uint64_t f64_bits(double v)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    uint64_t b;
    memcpy(&b, &v, sizeof b);
    return b;
#endif
}
__host__ __device__ __forceinline__ double f64_of(uint64_t b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double v;
    memcpy(&v, &b, sizeof v);
    return v;
#endif
}
__host__ __device__ __forceinline__ uint32_t f32_bits(float v)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(v);
#else
    uint32_t b;
    memcpy(&b, &v, sizeof b);
    return b;
#endif
}
__host__ __device__ __forceinline__ float f32_of(uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float v;
    memcpy(&v, &b, sizeof v);
    return v;
#endif
}

// The pair of a double in integer arithmetic, where both parts are normal
// floats: the FP64 unit, at 1/64 of the FP32 rate, takes four operations a
// value, which kept it half busy in K1 (256^3: 230 -> 209 us; 300^3: 679 -> 569).
// The values are those of df64(double); an exact tie between two leading
// floats may split the other way, to the same sum.  (The way back, done
// likewise, made K5 slower: 196 -> 206 us.)
__host__ __device__ __forceinline__ df64 df64_split(double d)
{
    const uint64_t b = f64_bits(d);
    const uint32_t w = (uint32_t)(b >> 32), sign = w & 0x80000000u, e = (w >> 20) & 0x7ffu;
    if (e - 950u < 199u) {
        // hi: the leading 24 bits, rounded; lo: the 29 bits below, as a signed
        // count of units of 2^(e - 1075)
        const int r = (int)((uint32_t)b << 3) >> 3;
        const uint32_t h = (uint32_t)((b + (1ull << 28)) >> 29) - (896u << 23);
        return {f32_of(h | sign), (float)r * f32_of((e - 948u) << 23 | sign)};
    }
    if ((b << 1) == 0) return {f32_of(sign), 0.0f};
    return df64(d);
}

// The real type an API buffer holds for arithmetic type T (df64 solves read
// and write FP64 arrays).
template <typename T>
struct IoReal {
    using type = T;
    static __host__ __device__ __forceinline__ T in(T v) { return v; }
    static __host__ __device__ __forceinline__ T out(T v) { return v; }
};
template <>
struct IoReal<df64> {
    using type = double;
    static __host__ __device__ __forceinline__ df64 in(double v) { return df64_split(v); }
    static __host__ __device__ __forceinline__ double out(df64 v) { return v.to_double(); }
};

}  // namespace isofft
