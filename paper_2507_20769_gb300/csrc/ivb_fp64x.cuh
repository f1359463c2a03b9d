// ivb_fp64x.cuh -- directed-rounding primitives built for a narrow FP64 pipe
// (GB300: one FP64 warp instruction per 64 cycles per SM sub-partition, integer /
// FP32 / MUFU pipes many times wider).
//
// Reciprocal, quotient, square root, exp and log in fixed point on the integer
// pipes (ivb_fixed.cuh) with their tables, and the inputs that take another
// path: results that are not normal doubles go to the CUDA intrinsics, exp
// beyond |x| = 700 and log of subnormals to CUDA's functions widened by two
// steps, and log next to 1, where the result needs more than 64 bits after
// the point, to a table-driven evaluation in FP64.
#pragma once
#ifndef __CUDACC_RTC__
#include <cstdint>
#endif

namespace ivb {

__device__ __forceinline__ float rcp_approx_f(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_approx_f(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

}  // namespace ivb

#include "ivb_fixed.cuh"

namespace ivb {

// tables, in device memory of this module (filled by init_math_tables, or
// copied from the library's tables into a tape-specialised module)
constexpr int kNearTab = 64;
struct NearEntry { double c, hi, lo; };        // centre c_j of [1 + j/2048, 1 + (j+1)/2048), -log(c_j) as hi + lo
struct MathTables {
    fx64 exp[kExpTab];         // 2^(j/512) in units of 2^-62
    LogEntry log[kLogTab];
    NearEntry near1[kNearTab]; // j = -32 .. 31 around 1 (j < 0: the interval's upper half, halved)
};
#if defined(__CUDACC_RTC__) && defined(IVB_JIT_EXTERN_TABLES)
extern __device__ MathTables g_math;   // defined by the kernel unit of a segmented module
#elif defined(__CUDACC_RTC__)
__device__ MathTables g_math;          // run-time compiled module: filled from the library's copy
#else
static __device__ MathTables g_math;
#endif

// Slow paths out of line: inlined, the compiler would start parts of them
// speculatively on the fast path, which costs FP64 issue slots every call.
static __device__ __noinline__ double rcp_slow(double y, bool up) { return up ? __drcp_ru(y) : __drcp_rd(y); }
static __device__ __noinline__ double div_slow(double x, double y, bool up) { return up ? __ddiv_ru(x, y) : __ddiv_rd(x, y); }
static __device__ __noinline__ double sqrt_slow(double x, bool up) { return up ? __dsqrt_ru(x) : __dsqrt_rd(x); }
static __device__ __noinline__ double exp_slow(double x) { return exp(x); }
static __device__ __noinline__ double log_slow(double x) { return log(x); }

__device__ __forceinline__ bool sign_of(double x) { return bits(x) < 0; }
__device__ __forceinline__ double with_sign(fx64 mag, bool neg) {
    return from_bits((long long)(mag | (neg ? 0x8000000000000000ULL : 0ULL)));
}

// correctly rounded 1/y toward -inf (up = false) or +inf, y != 0, finite or infinite
__device__ __forceinline__ double rcp_dir(double y, bool up) {
    if (!rcp_fits(y)) return rcp_slow(y, up);
    const bool neg = sign_of(y);
    return with_sign(rcp_mag(y, up != neg), neg);
}

// correctly rounded x/y, x and y finite, y != 0
__device__ __forceinline__ double div_dir(double x, double y, bool up) {
    const bool neg = sign_of(x) != sign_of(y);
    if ((bits(x) << 1) == 0) return with_sign(0, neg);     // exact: +-0
    if (!div_fits(x, y)) return div_slow(x, y, up);
    return with_sign(div_mag(x, y, rcp62(sig53(y)), up != neg), neg);
}

// correctly rounded sqrt(x), x >= 0
__device__ __forceinline__ double sqrt_dir(double x, bool up) {
    return sqrt_fits(x) ? from_bits((long long)sqrt_mag(x, up)) : sqrt_slow(x, up);
}

// double whose value is the integer k (|k| < 2^31), assembled on the integer
// pipe: sign, biased exponent 1023 + floor(log2 |k|) from the leading-zero
// count, and |k| shifted under the hidden bit (exact)
__device__ __forceinline__ double int_to_double(int k) {
    const unsigned a = k < 0 ? 0u - (unsigned)k : (unsigned)k;
    const int msb = 31 - __clz((int)a);                       // a > 0: position of the leading one
    const unsigned long long mant = ((unsigned long long)a << (52 - msb)) & 0x000FFFFFFFFFFFFFULL;
    const unsigned long long b = ((unsigned long long)(k < 0) << 63) |
                                 ((unsigned long long)(1023 + msb) << 52) | mant;
    return from_bits(a != 0u ? (long long)b : 0LL);
}

// float nearest to a double v with 2^-126 <= |v| < 2^127 (ties away from
// zero), 0 for smaller |v|; integer pipe only
__device__ __forceinline__ float f32_near(double v) {
    const long long b = bits(v);
    const int E = (int)((b >> 52) & 0x7FF);
    const long long m = (b & 0x7FFFFFFFFFFFFFFFLL) + (1LL << 28);   // round the 29 dropped bits
    const int fb = (int)((m >> 29) - ((long long)(1023 - 127) << 23));
    return __int_as_float(E > 1023 - 127 ? (fb | (int)((b >> 32) & 0x80000000)) : 0);
}
// log(x) for |log x| < 2^-7, error below 1.5 ulp of the result. With y = x,
// r = y c_j - 1 (exact for the two intervals next to 1, where c = 1; |r| <= 2^-11):
// log1p(r) = r + r^2 P(r), P = -1/2 + r/3 - r^2/4 + r^3/5, relative truncation
// below 2^-57 next to 1. delta = r^2 (-1/4 + r/5) is <= 0 and below 2^-22 in
// magnitude, so it goes on the FP32 pipe (its error reaches the result
// multiplied by r^2), and C = -1/2 + delta is assembled exactly on the integer
// pipe from delta cut to units of 2^-53: P = r/3 + C, one FP64 fma.
static __device__ __noinline__ double log_near1(double x) {
    const int j = (int)((bits(x) & 0x000FFFFFFFFFFFFFLL) >> 41);      // top 11 mantissa bits
    const NearEntry T = g_math.near1[(j + kNearTab / 2) & (kNearTab - 1)];
    const double r = __fma_rn(x, T.c, -1.0);
    const float rf = f32_near(r);
    const float delta = __fmul_rn(__fmul_rn(rf, rf), __fmaf_rn(rf, 0.2f, -0.25f));
    const int db = __float_as_int(delta) & 0x7FFFFFFF;
    const int sh = (db >> 23) - 127 + 30;              // |delta| = M 2^(sh - 53), M of 24 bits
    const long long M = (long long)((db & 0x7FFFFF) | 0x800000);
    const long long D = db == 0 ? 0LL : (sh >= 0 ? (M << sh) : (sh > -40 ? (M >> -sh) : 0LL));
    const double C = from_bits((long long)0xBFE0000000000000ULL | D);   // -(1/2 + D 2^-53)
    const double P = __fma_rn(r, 1.0 / 3.0, C);
    return T.hi + (__fma_rn(r * r, P, r) + T.lo);
}

// exp and log rounded outward (up: toward +inf); log: x > 0
__device__ __forceinline__ double exp_dir(double x, bool up) {
    if (exp_fits(x)) return from_bits((long long)exp_mag(x, g_math.exp, up));
    const double y = exp_slow(x);
    return up ? next_up(next_up(y)) : next_dn(next_dn(y));
}
__device__ __forceinline__ double log_dir(double x, bool up) {
    double y;
    const bool fits = log_fits(x);
    if (fits && log_val(x, g_math.log, up ? FX_UP : FX_DOWN, &y)) return y;
    y = fits ? log_near1(x) : log_slow(x);
    return up ? next_up(next_up(y)) : next_dn(next_dn(y));
}

// round to nearest (the point gradients): quotients, reciprocals and roots
// correctly rounded, exp within 0.51 and log within 0.52 units of the last place
// (measured 0.505 and 0.52, CUDA's 0.85 and 0.53); other results than normal
// doubles, and log closer to 1, from CUDA's functions
static __device__ __noinline__ double div_slow_rn(double x, double y) { return __ddiv_rn(x, y); }
static __device__ __noinline__ double sqrt_slow_rn(double x) { return __dsqrt_rn(x); }
__device__ __forceinline__ double rcp_rn(double y) {
    return rcp_fits(y) ? with_sign(rcp_near(y), sign_of(y)) : div_slow_rn(1.0, y);
}
__device__ __forceinline__ double div_rn(double x, double y) {
    return div_fits(x, y) ? with_sign(div_near(x, y), sign_of(x) != sign_of(y)) : div_slow_rn(x, y);
}
__device__ __forceinline__ double sqrt_rn(double x) {
    return sqrt_fits(x) ? from_bits((long long)sqrt_near(x)) : sqrt_slow_rn(x);
}
__device__ __forceinline__ double exp_rn(double x) {
    return exp_fits(x) ? from_bits((long long)exp_near(x, g_math.exp)) : exp_slow(x);
}
__device__ __forceinline__ double log_rn(double x) {
    double y;
    return log_fits(x) && log_val(x, g_math.log, FX_NEAR, &y) ? y : log_slow(x);
}

}  // namespace ivb
