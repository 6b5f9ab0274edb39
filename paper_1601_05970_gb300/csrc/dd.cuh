// Double-float numbers: the unevaluated sum hi + lo of two FP32 numbers
// with |lo| <= ulp(hi)/2, about 48 significant bits (relative rounding
// near 2^-47, some 7e-15).
//
// The arithmetic is built from the error-free transformations of Dekker
// ("A floating-point technique for extending the available precision",
// 1971) and Knuth (TAOCP vol. 2, 4.2.2):
//   TwoSum(a, b)     = (s, e) with s = fl(a + b) and a + b = s + e exactly;
//   FastTwoSum(a, b) = the same in three operations when |a| >= |b|;
//   TwoProd(a, b)    = (p, e) with p = fl(a b) and a b = p + e exactly,
//                      e = fma(a, b, -p).
// Addition is Dekker's: TwoSum of the high parts, the low parts added to
// the error term, renormalised by FastTwoSum; its error is a few units of
// 2^-47 of |a| + |b|, which suits an FFT (whose rounding error scales with
// the norm of its input anyway). Multiplication is TwoProd plus the cross
// terms.
//
// The residual pass of the mixed-precision path runs its FFTs in this
// format: GB300 executes FP32 at many times its FP64 rate, and the residual
// only needs accuracy well below the CG roundoff floor (1e-13 of ||sigma||).
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

namespace fftg {

struct __align__(8) dd {
    float hi, lo;
    dd() = default;
    __host__ __device__ constexpr dd(float h, float l) : hi(h), lo(l) {}
    // nearest double-float to v: hi = fl32(v), lo = fl32(v - hi)
    __host__ __device__ constexpr dd(double v) : hi((float)v), lo((float)(v - (double)(float)v)) {}
    __host__ __device__ constexpr explicit dd(int v) : hi((float)v), lo(0.0f) {}
    __host__ __device__ constexpr explicit operator double() const { return (double)hi + (double)lo; }
    __host__ __device__ constexpr explicit operator float() const { return hi + lo; }
};

// Round-to-nearest FP32 primitives that the compiler may not fuse or
// reorder: the CUDA intrinsics on the device, plain IEEE float arithmetic
// (and std::fma) on the host, where the arithmetic is tested.
__host__ __device__ __forceinline__ float dd_add(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    volatile float s = a + b;
    return s;
#endif
}
__host__ __device__ __forceinline__ float dd_sub(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fsub_rn(a, b);
#else
    volatile float s = a - b;
    return s;
#endif
}
__host__ __device__ __forceinline__ float dd_mul(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    volatile float s = a * b;
    return s;
#endif
}
__host__ __device__ __forceinline__ float dd_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fma(a, b, c);
#endif
}

// TwoSum: s + e = a + b exactly
__host__ __device__ __forceinline__ dd dd_two_sum(float a, float b) {
    const float s = dd_add(a, b);
    const float bb = dd_sub(s, a);
    const float e = dd_add(dd_sub(a, dd_sub(s, bb)), dd_sub(b, bb));
    return dd(s, e);
}

// FastTwoSum: s + e = a + b exactly when |a| >= |b|
__host__ __device__ __forceinline__ dd dd_fast_two_sum(float a, float b) {
    const float s = dd_add(a, b);
    return dd(s, dd_sub(b, dd_sub(s, a)));
}

// TwoProd: p + e = a b exactly
__host__ __device__ __forceinline__ dd dd_two_prod(float a, float b) {
    const float p = dd_mul(a, b);
    return dd(p, dd_fma(a, b, -p));
}

__host__ __device__ __forceinline__ dd operator+(dd a, dd b) {
    const dd s = dd_two_sum(a.hi, b.hi);
    return dd_fast_two_sum(s.hi, dd_add(s.lo, dd_add(a.lo, b.lo)));
}

__host__ __device__ __forceinline__ dd operator-(dd a) { return dd(-a.hi, -a.lo); }

__host__ __device__ __forceinline__ dd operator-(dd a, dd b) { return a + (-b); }

__host__ __device__ __forceinline__ dd operator*(dd a, dd b) {
    const dd p = dd_two_prod(a.hi, b.hi);
    float e = dd_fma(a.hi, b.lo, p.lo);
    e = dd_fma(a.lo, b.hi, e);
    return dd_fast_two_sum(p.hi, e);
}

__host__ __device__ __forceinline__ dd& operator+=(dd& a, dd b) { return a = a + b; }

__host__ __device__ __forceinline__ bool operator>(dd a, dd b) {
    return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo);
}
__host__ __device__ __forceinline__ bool operator<(dd a, dd b) { return b > a; }

// Conversions by integer arithmetic. The device converts between FP32 and FP64
// at about its FP64 rate (1/74 of FP32). These give the bits of the plain
// casts, which they use for the exponents they leave out (subnormal, out of
// range). The pass that splits an FP64 field into double-floats: 1.29 -> 1.19
// ms at 243^3, 77 -> 61 us for 32 cells of 27^3 (nine components of finite
// strain, where registers bound it, lose 10 % and keep the casts).
__host__ __device__ __forceinline__ unsigned long long bits_of(double v) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long u;
    std::memcpy(&u, &v, 8);
    return u;
#endif
}
__host__ __device__ __forceinline__ float float_of_bits(unsigned b) {
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float f;
    std::memcpy(&f, &b, 4);
    return f;
#endif
}

// |v| rounded to nearest even at FP32's last bit, as the FP64 pattern's upper
// part: exponent (11 bits) and 23 bits. For the sign bit cleared.
__host__ __device__ __forceinline__ unsigned long long round_to_f32(unsigned long long mag) {
    return (mag + 0x0fffffffull + ((mag >> 29) & 1ull)) >> 29;
}

// (float)v
__host__ __device__ __forceinline__ float f32_of(double v) {
    const unsigned long long u = bits_of(v), mag = u & 0x7fffffffffffffffull;
    const unsigned e = (unsigned)(mag >> 52), sign = (unsigned)(u >> 32) & 0x80000000u;
    if (e - 897u > 1150u - 897u) return mag ? (float)v : float_of_bits(sign);
    return float_of_bits(((unsigned)round_to_f32(mag) - (896u << 23)) | sign);
}

// dd(v): hi = (float)v, lo = (float)(v - hi). The remainder v - hi is an
// integer of at most 29 bits in units of v's last place.
__host__ __device__ __forceinline__ dd dd_split(double v) {
    const unsigned long long u = bits_of(v), mag = u & 0x7fffffffffffffffull;
    const unsigned e = (unsigned)(mag >> 52), sign = (unsigned)(u >> 32) & 0x80000000u;
    if (e - 949u > 1149u - 949u) return mag ? dd(v) : dd(float_of_bits(sign), 0.0f);
    const unsigned long long r = round_to_f32(mag);
    const int rem = (int)((unsigned)mag & 0x1fffffffu) - (int)((unsigned)(r - (mag >> 29)) << 29);
    const float hi = float_of_bits(((unsigned)r - (896u << 23)) | sign);
    return dd(hi, dd_mul((float)(sign ? -rem : rem), float_of_bits((e - 948u) << 23)));
}

#ifdef __CUDACC__
// 1/sqrt(x) for the per-frequency factors of Ghat (FP64 rsqrt, rounded)
__device__ __forceinline__ dd rsqrt_t(dd x) { return dd(rsqrt((double)x)); }
#endif

}  // namespace fftg
