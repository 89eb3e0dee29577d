// FP64 elementary functions of the property paths.  The FP64 pipe is their
// scarce unit (2 operations per clock per SM on GB300), so the usual argument
// ranges are computed on the integer pipe (pr_int64.cuh); what they leave goes
// to the forms here, or to CUDA's functions:
//   rcp, div, sqrt   normal operands and results;
//   exp              |x| < 64 (else CUDA's exp);
//   expm1            2^-7 <= |x| < 64 (smaller: Tang's form below);
//   log, log1p       where |ln| is at least 2^-5 (nearer zero: Tang's form);
//   pow_neg, cbrt    x^-b for a constant b in (0, 1), x^(1/3), normal x > 0 (cbrt: x >= 0).
// Tang's table-driven forms (P. T. P. Tang, ACM TOMS 15 (1989) 144-157 and 16
// (1990) 378-400), with FP64 operations:
// exp: 64 table points: x = (64 m + j) ln2/64 + r, |r| <= ln2/128, exp(x) =
// 2^m 2^(j/64) e^r, the reduction in double-double by FMA, e^r - 1 by its
// Taylor polynomial to r^7 (expm1, whose result can be of the size of r),
// 2^(j/64) as a double-double table.
// log: F = 1 + j/128 nearest the significand m: ln x = e ln2 + ln F + ln(1 + r),
// r = (m - F)/F (m - F exact; 1/F from a table and one correction step),
// ln(1 + r) by its Taylor polynomial to r^8 (|r| <= 1/256).
// Errors in units in the last place: rcp, div and sqrt within 0.51 (2^-60 before
// the rounding); against quad precision, 2 M arguments a range: exp 0.59 (the
// argument's 64 bits at |x| near 64; 0.51 below 1), log and log1p 0.60 in the
// integer form (1.2 and 1.5 in Tang's near zero), expm1 0.64 from 2^-5, 1.08
// from 2^-7 to 2^-5 (the absolute error of 2^-60 against a small result), 1.35
// below.  Tests (tests/test_gpu_math64.py): within 1.5.
#pragma once

#include <cuda_runtime.h>

#include "math64_tables.h"
#include "pr_int64.cuh"

namespace m64 {

// round-to-nearest integer of x * 64/ln2 via the 1.5 * 2^52 shifter
constexpr double kShift = 6755399441055744.0;

// e^r - 1 for |r| <= ln2/128: the truncation is below 5e-18 of it
__device__ __forceinline__ double expm1_small_rel(double r)
{
    const double r2 = r * r;
    double q = fma(r, 1.0 / 5040.0, 1.0 / 720.0);
    q = fma(q, r, 1.0 / 120.0);
    q = fma(q, r, 1.0 / 24.0);
    q = fma(q, r, 1.0 / 6.0);
    q = fma(q, r, 0.5);
    return fma(q, r2, r);
}

// e^x - 1 for |x| < 512: the 1 taken off before the scaled table value is
// rounded, so that small x keep their relative accuracy
static __device__ __noinline__ double expm1_tang(double x)
{
    const double t = fma(x, k64OverLn2, kShift);
    const double kd = t - kShift;
    const int k = __double2loint(t);
    double r = fma(-kd, kLn2Over64Hi, x);
    r = fma(-kd, kLn2Over64Lo, r);
    const double p = expm1_small_rel(r);
    const int j = k & 63, m = k >> 6;
    if (k == 0) return p;
    const double s = __hiloint2double((1023 + m) << 20, 0);   // 2^m
    const double th = __ldg(&kExp2Hi[j]) * s, tl = __ldg(&kExp2Lo[j]) * s;
    // 2^m 2^(j/64) (1 + p) - 1 = (th - 1) + (th p + tl); th - 1 is exact while th is within [1/2, 2]
    return (th - 1.0) + fma(th, p, tl);
}

// ln(1 + r) for |r| <= 1/256, to the r^8 term (the truncation is below
// 2^-64 / 9 of r: near x = 1 the logarithm is of the size of r)
__device__ __forceinline__ double log1p_small(double r)
{
    const double r2 = r * r;
    double q = fma(r, -1.0 / 8.0, 1.0 / 7.0);
    q = fma(q, r, -1.0 / 6.0);
    q = fma(q, r, 0.2);
    q = fma(q, r, -0.25);
    q = fma(q, r, 1.0 / 3.0);
    q = fma(q, r, -0.5);
    return fma(q, r2, r);
}

// ln x for finite positive normal x
static __device__ __noinline__ double log_tang(double x)
{
    const int hx = __double2hiint(x), lx = __double2loint(x);
    const int ex = (hx >> 20) & 0x7FF;
    if (ex == 0 || ex == 0x7FF || hx < 0) return ::log(x);
    // significand m in [1, 2); j: its leading 7 fraction bits, rounded
    const double m = __hiloint2double((hx & 0x000FFFFF) | 0x3FF00000, lx);
    const int j = ((hx & 0x000FFFFF) + (1 << 12)) >> 13;       // 0..128
    const double F = __hiloint2double(0x3FF00000 + (j << 13), 0);   // 1 + j/128 (2 for j = 128)
    // r = (m - F) / F: the product with the rounded 1/F, then one correction
    // step from the exact residual (m - F) - r F
    const double f = m - F, iF = __ldg(&kInvF[j]);
    double r = f * iF;
    r = fma(fma(-r, F, f), iF, r);
    const double lp = log1p_small(r);
    const double e = (double)(ex - 1023);
    const double hi = fma(e, kLn2Hi, __ldg(&kLogFHi[j]));
    const double lo = fma(e, kLn2Lo, __ldg(&kLogFLo[j]));
    return hi + (lp + lo);
}

// ln(1 + z) for z > -1: ln u of the rounded u = 1 + z, plus the rounding
// error of u over u (a tiny correction, taken with a single-precision 1/u)
static __device__ __noinline__ double log1p_tang(double z)
{
    const double u = 1.0 + z;
    const double c = z - (u - 1.0);
    return log_tang(u) + c * (double)__frcp_rn((float)u);
}

// ------------------------------------------------ integer-pipe forms
// the general operations, out of line: reached by zeros, infinities, NaN,
// subnormals and results near the ends of the range
static __device__ __noinline__ double slow_div(double a, double b) { return a / b; }
static __device__ __noinline__ double slow_sqrt(double x) { return ::sqrt(x); }
static __device__ __noinline__ double slow_exp(double x) { return ::exp(x); }
static __device__ __noinline__ double slow_expm1(double x) { return ::expm1(x); }
static __device__ __noinline__ double slow_pow(double x, double y) { return ::pow(x, y); }

__device__ __forceinline__ double rcp(double x)
{
    const uint64_t b = i64::bits(x);
    const uint32_t e = i64::expo(b);
    if (e - 1u >= 2044u) return slow_div(1.0, x);
    const uint64_t r = i64::pack_bits(i64::rcp_m(i64::signif(b)), 1022 - (int)e);
    return i64::from_bits(r | (b & 0x8000000000000000ull));
}

__device__ __forceinline__ double div(double a, double b)
{
    const uint64_t ba = i64::bits(a), bb = i64::bits(b);
    const uint32_t ea = i64::expo(ba), eb = i64::expo(bb);
    if (ea - 1u >= 2046u || eb - 1u >= 2046u || ea - eb + 1000u > 2000u) return slow_div(a, b);
    uint64_t q = i64::mulhi(i64::signif(ba), i64::rcp_m(i64::signif(bb)));   // in (2^62, 2^64)
    int e = (int)ea - (int)eb;
    if (!(q >> 63)) {
        q <<= 1;
        --e;
    }
    return i64::from_bits(i64::pack_bits(q, e) | ((ba ^ bb) & 0x8000000000000000ull));
}

__device__ __forceinline__ double sqrt(double x)
{
    const uint64_t b = i64::bits(x);
    const uint32_t e = (uint32_t)(b >> 52);   // with the sign bit: negative x leaves the range
    if (e - 1u >= 2046u) return slow_sqrt(x);
    // x = X 2^(2 h), X in [1/4, 1): the significand halved (e even: an odd power of two) or quartered
    const uint64_t X = i64::signif(b) >> (e & 1u);
    const uint64_t s = i64::mulhi(X, i64::rsqrt_m(X)) << 1;
    const int h = ((int)e - 1022 + (int)(e & 1u)) / 2;   // even numerator
    return i64::from_bits(i64::pack_bits(s, h - 1));
}

// 2^-(n + F / 2^64), rounded; |n| <= 1000
__device__ __forceinline__ double pack_exp2_neg(int n, uint64_t F)
{
    const uint64_t r = i64::exp2_neg(F);   // units 2^-63, in (2^62, 2^63]
    const uint64_t q = (r >> 10) + ((r >> 9) & 1u);
    return i64::from_bits(q + ((uint64_t)(uint32_t)(1021 - n) << 52));
}

// -x log2(e) = n + F / 2^64 for 2^-60 <= |x| < 64 (biased exponent e)
__device__ __forceinline__ int exp_arg(uint64_t b, uint32_t e, uint64_t &F)
{
    const uint64_t p = i64::mulhi(i64::signif(b), kI64Log2E);   // |x| log2 e = p 2^(e - 1023 - 62)
    const int s = 1085 - (int)e;                                   // 57..: bits of p below the point
    int n = 0;
    if (s >= 64) {
        F = p >> (s - 64);
    } else {
        F = p << (64 - s);
        n = (int)(p >> s);
    }
    if (!(b >> 63)) {   // x > 0: -(n + F)
        n = -n - (F != 0);
        F = 0 - F;
    }
    return n;
}

__device__ __forceinline__ double exp(double x)
{
    const uint64_t b = i64::bits(x);
    const uint32_t e = i64::expo(b);
    if (e - 963u >= 66u) return slow_exp(x);   // |x| outside [2^-60, 64)
    uint64_t F;
    const int n = exp_arg(b, e, F);
    return pack_exp2_neg(n, F);
}

__device__ __forceinline__ double expm1(double x)
{
    const uint64_t b = i64::bits(x);
    const uint32_t e = i64::expo(b);
    if (e - 1016u >= 13u) return e >= 1029u ? slow_expm1(x) : expm1_tang(x);   // |x| outside [2^-7, 64)
    uint64_t F;
    const int n = exp_arg(b, e, F);
    const uint64_t r = i64::exp2_neg(F);   // e^x = r 2^-(63 + n)
    uint64_t d;
    int ex;   // |result| = d 2^(ex - 63)
    if (b >> 63) {   // n >= 0: 1 - e^x
        d = 0x8000000000000000ull - (n < 64 ? r >> n : 0);
        ex = 0;
    } else {         // n < 0: e^x - 1, in units of 2^(-63 - n)
        d = r - (-n < 64 ? 0x8000000000000000ull >> -n : 0);
        ex = -n;
    }
    const int z = __clzll((long long)d);
    return i64::from_bits(i64::pack_bits(d << z, ex - z) | (b & 0x8000000000000000ull));
}

// ln of m 2^E with m = M / 2^63 in [1, 2); |ln| at least about 2^-6
__device__ __forceinline__ double ln_parts(uint64_t M, int E)
{
    uint64_t l = i64::log2_m(M);
    const bool neg = E < 0;
    if (neg) {   // |E + l| = (-E - 1) + (1 - l)
        E = -E - (l != 0);
        l = 0 - l;
    }
    // E + l as a normalised 64-bit number v 2^(k - 63)
    const int k = E ? 31 - __clz(E) : -1 - __clzll((long long)l);
    const uint64_t v = E ? ((uint64_t)(uint32_t)E << (63 - k)) | (l >> (k + 1)) : l << (-1 - k);
    uint64_t q = i64::mulhi(v, kI64Ln2);   // in (2^62, 2^64)
    int e = k;
    if (!(q >> 63)) {
        q <<= 1;
        --e;
    }
    return i64::from_bits(i64::pack_bits(q, e) | (neg ? 0x8000000000000000ull : 0));
}

__device__ __forceinline__ double log(double x)
{
    const uint64_t b = i64::bits(x);
    const uint32_t e = (uint32_t)(b >> 52);
    // x within [1 - 2^-5, 1 + 2^-5), or not a positive normal number
    const uint64_t d = b - 0x3FEF000000000000ull;
    if (e - 1u >= 2046u || d < 0x0001800000000000ull) return log_tang(x);
    return ln_parts(i64::signif(b), (int)e - 1023);
}

__device__ __forceinline__ double log1p(double z)
{
    const uint64_t b = i64::bits(z);
    const uint32_t e = (uint32_t)(b >> 52);
    if (e - 1018u >= 57u) return log1p_tang(z);   // z outside [2^-5, 2^52)
    // 1 + z, exact in 64 bits
    uint64_t M = i64::signif(b);
    int E = (int)e - 1023;
    if (E < 0) {
        M = 0x8000000000000000ull + (M >> -E);
        E = 0;
    } else {
        const uint64_t s = M + (0x8000000000000000ull >> E);
        const bool carry = s < M;
        M = carry ? (s >> 1) | 0x8000000000000000ull : s;
        E += carry;
    }
    return ln_parts(M, E);
}

// x^-b in units of 2^-64 for the bits of a normal x with x^-b below 1, b = B / 2^64
__device__ __forceinline__ uint64_t pow_frac_fixed(uint64_t bx, uint64_t B)
{
    const uint32_t E = (uint32_t)(bx >> 52) - 1023u;   // x >= 1: E >= 0
    const uint64_t w0 = i64::wide(i64::lo32(B), E), w1 = i64::wide(i64::hi32(B), E) + (w0 >> 32);
    const uint64_t F = (w1 << 32) | i64::lo32(w0);
    const uint64_t G = F + i64::mulhi(i64::log2_m(i64::signif(bx)), B);
    const uint32_t n = (uint32_t)(w1 >> 32) + (G < F);
    return (i64::exp2_neg(G) << 1) >> n;
}

// x^-b (or, NEG = false, x^b) for a positive normal x and b = B / 2^64 in (0, 1)
template <bool NEG>
__device__ __forceinline__ double pow_frac(double x, uint64_t B)
{
    const uint64_t bx = i64::bits(x);
    const uint32_t e = (uint32_t)(bx >> 52);
    if (e - 1u >= 2046u) return slow_pow(x, (NEG ? -5.421010862427522e-20 : 5.421010862427522e-20) * (double)B);
    // b log2 x = b E + b l
    const int E = (int)e - 1023;
    const uint32_t a = (uint32_t)(E < 0 ? -E : E);
    const uint64_t w0 = i64::wide(i64::lo32(B), a), w1 = i64::wide(i64::hi32(B), a) + (w0 >> 32);
    uint64_t F = (w1 << 32) | i64::lo32(w0);
    int n = (int)(w1 >> 32);
    if (E < 0) {
        n = -n - (F != 0);
        F = 0 - F;
    }
    uint64_t G = F + i64::mulhi(i64::log2_m(i64::signif(bx)), B);
    n += G < F;
    if (!NEG) {
        n = -n - (G != 0);
        G = 0 - G;
    }
    return pack_exp2_neg(n, G);
}
__device__ __forceinline__ double pow_neg(double x, uint64_t B) { return pow_frac<true>(x, B); }
__device__ __forceinline__ double cbrt(double x) { return pow_frac<false>(x, 0x5555555555555555ull); }   // x >= 0

}  // namespace m64
