// Element operations of the scheme code (mhd_math.cuh), written as functions so that the
// arithmetic reads the same for float and double and states its roundings: fused
// multiply-adds are explicit, and region choices are selections rather than branches
// (comparisons give a mask, sel() picks).
//
// Helpers used by the scheme code for R = float, double:
//   fma_(a, b, c) = a * b + c rounded once      sel(m, a, b) = m ? a : b
//   mul_(a, b) = a * b, never fused
//   nonneg_, le_mag_, greater_ ... -> mask       mand / mor / mnot on masks
//   rabs, rdiv (quotient), rsqrt_ (square root), rcp_ (reciprocal), fmax_ / fmin_ (larger / smaller
//   value)
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#ifndef MHD_HD
#define MHD_HD __host__ __device__ __forceinline__
#endif

namespace mhd {

MHD_HD float fma_(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return fmaf(a, b, c);
#endif
}
MHD_HD double fma_(double a, double b, double c) {
#ifdef __CUDA_ARCH__
    return __fma_rn(a, b, c);
#else
    return fma(a, b, c);
#endif
}

// a * b rounded on its own: never fused into a neighbouring addition by the compiler, so
// that every kernel that evaluates the same expression rounds it the same way
MHD_HD float mul_(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
MHD_HD double mul_(double a, double b) {
#ifdef __CUDA_ARCH__
    return __dmul_rn(a, b);
#else
    return a * b;
#endif
}

// Comparisons.  Double precision on the device: on the bits (doubles of one sign order as integers),
// off the FP64 pipe, whose 2 lanes per clock and SM bound every FP64 kernel and on which a comparison
// costs as much as a product; the integer pipe has 64 and is idle.  They give what the comparison of
// the values gives: the two zeros are equal, and a NaN compares false.
#ifdef __CUDA_ARCH__
constexpr long long kInfBits = 0x7ff0000000000000ll, kMagBits = 0x7fffffffffffffffll;
// bits of a double ordered as the values (and back); order0_: and the two zeros equal
__device__ __forceinline__ long long order_(long long i) { return i ^ (long long)((unsigned long long)(i >> 63) >> 1); }
__device__ __forceinline__ long long order0_(long long i) { return i < 0 ? (long long)0x8000000000000000ull - i : i; }
#endif
// x is a number
MHD_HD bool number_(float x) { return x == x; }
MHD_HD bool number_(double x) {
#ifdef __CUDA_ARCH__
    return (__double_as_longlong(x) & kMagBits) <= kInfBits;
#else
    return x == x;
#endif
}
// x >= 0; a <= b for two magnitudes (a not NaN, or b a number)
MHD_HD bool nonneg_(float x) { return x >= 0.0f; }
MHD_HD bool nonneg_(double x) {
#ifdef __CUDA_ARCH__
    const long long i = __double_as_longlong(x);
    return (unsigned long long)i <= (unsigned long long)kInfBits || (i << 1) == 0;   // (-0 is not below 0)
#else
    return x >= 0.0;
#endif
}
MHD_HD bool le_mag_(float a, float b) { return a <= b; }
MHD_HD bool le_mag_(double a, double b) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(a) <= __double_as_longlong(b);
#else
    return a <= b;
#endif
}
// x != 0; x > 0; a > b
MHD_HD bool nonzero_(float x) { return x != 0.0f; }
MHD_HD bool positive_(float x) { return x > 0.0f; }
MHD_HD bool greater_(float a, float b) { return a > b; }
MHD_HD bool nonzero_(double x) {
#ifdef __CUDA_ARCH__
    return (__double_as_longlong(x) << 1) != 0;
#else
    return x != 0.0;
#endif
}
MHD_HD bool positive_(double x) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)(__double_as_longlong(x) - 1) < (unsigned long long)kInfBits;
#else
    return x > 0.0;
#endif
}
MHD_HD bool greater_(double a, double b) {
#ifdef __CUDA_ARCH__
    const long long i = order0_(__double_as_longlong(a)), j = order0_(__double_as_longlong(b));
    return i > j && i <= kInfBits && j >= -kInfBits;
#else
    return a > b;
#endif
}
// a and b of the same sign and neither 0, without the product a b, which underflows where both are
// small (in single precision at 1e-19): the condition under which minmod_ below is not 0
MHD_HD bool same_sign_(float a, float b) { return (a > 0.0f && b > 0.0f) || (a < 0.0f && b < 0.0f); }
MHD_HD bool same_sign_(double a, double b) {
#ifdef __CUDA_ARCH__
    const long long i = __double_as_longlong(a), j = __double_as_longlong(b);
    return (i ^ j) >= 0 && (unsigned long long)((i & kMagBits) - 1) < (unsigned long long)kInfBits &&
           (unsigned long long)((j & kMagBits) - 1) < (unsigned long long)kInfBits;
#else
    return (a > 0.0 && b > 0.0) || (a < 0.0 && b < 0.0);
#endif
}
MHD_HD bool mand(bool a, bool b) { return a && b; }
MHD_HD bool mor(bool a, bool b) { return a || b; }
MHD_HD bool mnot(bool a) { return !a; }
template <typename R>
MHD_HD R sel(bool m, R a, R b) { return m ? a : b; }

// |x| (the sign of a zero result is +0; the scheme only compares magnitudes or divides
// them, so it never depends on that sign).  fabs lets the compiler fold |.| into the
// consuming instruction as an operand modifier instead of a compare and a select.
MHD_HD float rabs(float x) { return fabsf(x); }
MHD_HD double rabs(double x) { return fabs(x); }

// Square root and reciprocal.  Single precision on the device: the compiler's approximate square root,
// the hardware's approximate reciprocal (1 ulp).  Double precision on the device, from the hardware's
// 20-bit approximations (rsqrt.approx.ftz.f64, rcp.approx.ftz.f64), in two forms:
//
// rsqrt_near_, rcp_near_: within 0.509 and 0.507 ulp, five and three operations.
//   rcp:  e = 1 - x y, 1/x = y (1 + e + e^2 + O(e^3)), one step of third order (Householder);
//   sqrt: g = x y, h = y / 2 (on the exponent), r = 1/2 - g h, g' = g (1 + r), then the residual of
//         g' with the same h (Goldschmidt's and Newton's steps, as in P. Markstein's IA-64 and
//         Elementary Functions).
// rsqrt_, rcp_: correctly rounded, as the IEEE operations.  The near form is the right value or a
//   neighbour of it, and its residual, exact in one fused operation, decides (Tuckerman's test): the
//   value moves by one unit in the last place where the residual exceeds what half a unit makes,
//   x ulp(y) / 2 or g ulp(g), compared on the bits.
// Arguments outside [2^-900, 2^900] (0, denormals, infinities, NaN and negative ones among them) take
// the IEEE operation in both.
//
// The results of the scheme (primitive variables, predictor, CFL rates) take the correctly rounded
// form.  The face and edge solvers and their reverses, whose FP64 operations bound the double-precision
// step, take the near one: with the rounded form there the step of a 128^3 box takes 11.4 instead of
// 9.8 ms, and the error of a flux, an EMF or a cotangent is the same to four digits (HLLD flux, 1e4
// random faces, against extended precision: rms 0.640 units of 2^-53 of the largest component either
// way; 1.130 with IEEE operations in the form that preceded this one).
#ifdef __CUDA_ARCH__
static __device__ __noinline__ double sqrt_slow_(double x) { return sqrt(x); }
static __device__ __noinline__ double rcp_slow_(double x) { return 1.0 / x; }
// the argument is in the range of the fast forms (biased exponents 1023 - 900 to 1023 + 899)
__device__ __forceinline__ bool sqrt_range_(double x) { return (unsigned)__double2hiint(x) - (123u << 20) < (1800u << 20); }
__device__ __forceinline__ bool rcp_range_(double x) {
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) - (123u << 20) < (1800u << 20);
}
__device__ __forceinline__ double sqrt_fast_(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double g = __dmul_rn(x, y);
    const double h = __hiloint2double(__double2hiint(y) - (1 << 20), __double2loint(y));
    const double g1 = __fma_rn(g, __fma_rn(-g, h, 0.5), g);
    return __fma_rn(__fma_rn(-g1, g1, x), h, g1);
}
__device__ __forceinline__ double rcp_fast_(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double r = __fma_rn(-x, y, 1.0);
    return __fma_rn(y, __fma_rn(r, r, r), y);
}
#endif
MHD_HD float rsqrt_(float x) { return sqrtf(x); }
MHD_HD float rsqrt_near_(float x) { return sqrtf(x); }
MHD_HD double rsqrt_near_(double x) {
#ifdef __CUDA_ARCH__
    return sqrt_range_(x) ? sqrt_fast_(x) : sqrt_slow_(x);
#else
    return sqrt(x);
#endif
}
MHD_HD double rsqrt_(double x) {
#ifdef __CUDA_ARCH__
    if (!sqrt_range_(x)) return sqrt_slow_(x);
    const double g = sqrt_fast_(x);
    const long long b = __double_as_longlong(g), d = __double_as_longlong(__fma_rn(-g, g, x));
    // g times the unit in its last place, and times the one below it (a power of two has half)
    const long long up = b + (((b >> 52) - 1075) << 52), down = b + ((((b - 1) >> 52) - 1075) << 52);
    return __longlong_as_double(b + (d > up ? 1 : (d < 0 && (d & kMagBits) >= down ? -1 : 0)));
#else
    return sqrt(x);
#endif
}
MHD_HD float rcp_(float x) {
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / x;
#endif
}
MHD_HD float rcp_near_(float x) { return rcp_(x); }
MHD_HD double rcp_near_(double x) {
#ifdef __CUDA_ARCH__
    return rcp_range_(x) ? rcp_fast_(x) : rcp_slow_(x);
#else
    return 1.0 / x;
#endif
}
MHD_HD double rcp_(double x) {
#ifdef __CUDA_ARCH__
    if (!rcp_range_(x)) return rcp_slow_(x);
    const double y = rcp_fast_(x);
    const long long b = __double_as_longlong(y), d = __double_as_longlong(__fma_rn(-x, y, 1.0));
    const long long half = (__double_as_longlong(x) & kMagBits) + ((((b & kMagBits) >> 52) - 1076) << 52);
    return __longlong_as_double(b + ((d & kMagBits) > half ? (d < 0 ? -1 : 1) : 0));
#else
    return 1.0 / x;
#endif
}

// Quotient.  Single precision on the device: the hardware approximate division
// (__fdividef: a reciprocal and a multiply, within 2 ulp for divisors below 2^126 in
// magnitude, which every divisor of the scheme is); double precision and host code: the
// IEEE operation.
MHD_HD float rdiv(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fdividef(a, b);
#else
    return a / b;
#endif
}
MHD_HD double rdiv(double a, double b) { return a / b; }

// a / b from y, the reciprocal of b or a near one.  Double precision on the device: the product and one
// step on its residual (Markstein), rounded once like the quotient itself, where a y is rounded twice
// (and y's 0.507 ulp come on top); two operations more.  Single precision: the product.
MHD_HD float quot_(float a, float b, float y) { return a * y; }
MHD_HD double quot_(double a, double b, double y) {
#ifdef __CUDA_ARCH__
    const double q = __dmul_rn(a, y), q1 = __fma_rn(__fma_rn(-b, q, a), y, q);
    // (an infinite or zero y, an overflow: the product)
    return (__double2hiint(q1) & 0x7ff00000) != 0x7ff00000 ? q1 : q;
#else
    return a / b;
#endif
}

// x is finite (tested in its own precision: no conversion to double)
MHD_HD bool finite_(float x) { return isfinite(x); }
MHD_HD bool finite_(double x) { return isfinite(x); }

// Larger / smaller of two values; a NaN is passed over, as in fmaxf and fminf (a corner's speeds are
// NaN where its extrapolated density is negative: the others' decide then).
MHD_HD float fmax_(float a, float b) { return fmaxf(a, b); }
MHD_HD float fmin_(float a, float b) { return fminf(a, b); }
MHD_HD double fmax_(double a, double b) {
#ifdef __CUDA_ARCH__
    const bool p = order_(__double_as_longlong(a)) >= order_(__double_as_longlong(b));
    const double m = p ? a : b;
    return number_(m) ? m : (p ? b : a);
#else
    return fmax(a, b);
#endif
}
MHD_HD double fmin_(double a, double b) {
#ifdef __CUDA_ARCH__
    const bool p = order_(__double_as_longlong(a)) <= order_(__double_as_longlong(b));
    const double m = p ? a : b;
    return number_(m) ? m : (p ? b : a);
#else
    return fmin(a, b);
#endif
}

// max(a, b, c, d, 0) and min(a, b, c, d, 0), NaN passed over.  Single precision: two three-input
// instructions (sm_100 and later); double precision: on the bits, as above (of values among which 0 is,
// the largest signed integer is the largest value; the smallest value is the largest with its sign
// turned; a NaN whose sign makes it the largest counts as 0).
#ifdef __CUDA_ARCH__
__device__ __forceinline__ long long max0_bits_(long long a, long long b, long long c, long long d) {
    auto num = [](long long i) { return i > kInfBits ? 0ll : i; };
    return max(max(max(num(a), num(b)), max(num(c), num(d))), 0ll);
}
#endif
MHD_HD float max0_(float a, float b, float c, float d) {
#ifdef __CUDA_ARCH__
    float r;
    asm("{\n .reg .f32 t;\n max.ftz.f32 t, %1, %2, %3;\n max.ftz.f32 %0, t, %4, %5;\n}\n"
        : "=f"(r)
        : "f"(a), "f"(b), "f"(c), "f"(d), "f"(0.0f));
    return r;
#else
    return fmaxf(fmaxf(fmaxf(a, b), fmaxf(c, d)), 0.0f);
#endif
}
MHD_HD float min0_(float a, float b, float c, float d) {
#ifdef __CUDA_ARCH__
    float r;
    asm("{\n .reg .f32 t;\n min.ftz.f32 t, %1, %2, %3;\n min.ftz.f32 %0, t, %4, %5;\n}\n"
        : "=f"(r)
        : "f"(a), "f"(b), "f"(c), "f"(d), "f"(0.0f));
    return r;
#else
    return fminf(fminf(fminf(a, b), fminf(c, d)), 0.0f);
#endif
}
MHD_HD double max0_(double a, double b, double c, double d) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(max0_bits_(__double_as_longlong(a), __double_as_longlong(b), __double_as_longlong(c),
                                           __double_as_longlong(d)));
#else
    return fmax(fmax(fmax(a, b), fmax(c, d)), 0.0);
#endif
}
MHD_HD double min0_(double a, double b, double c, double d) {
#ifdef __CUDA_ARCH__
    const long long s = (long long)0x8000000000000000ull;
    return __longlong_as_double(max0_bits_(__double_as_longlong(a) ^ s, __double_as_longlong(b) ^ s,
                                           __double_as_longlong(c) ^ s, __double_as_longlong(d) ^ s) ^ s);
#else
    return fmin(fmin(fmin(a, b), fmin(c, d)), 0.0);
#endif
}

// minmod(a, b): the argument of smaller magnitude when both have the same sign, else 0, i.e.
// the median of a, b and 0 (double precision: 0 beside a NaN).
MHD_HD float minmod_(float a, float b) {
    return fminf(fmaxf(a, fminf(b, 0.0f)), fmaxf(b, 0.0f));
}
MHD_HD double minmod_(double a, double b) {
#ifdef __CUDA_ARCH__
    const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
    const long long ma = ia & kMagBits, mb = ib & kMagBits;
    const long long pick = ma <= mb ? ia : ib;
    return __longlong_as_double((ia ^ ib) < 0 || max(ma, mb) > kInfBits ? 0ll : pick);
#else
    return same_sign_(a, b) ? (fabs(a) <= fabs(b) ? a : b) : 0.0;
#endif
}

}  // namespace mhd
