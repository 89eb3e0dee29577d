// FP64 results from the integer and FP32 pipes.
//
// GB300 issues 2 FP64 operations per clock per SM and 64 or more 32-bit
// integer multiply-adds, so a 64 x 64-bit product (four IMAD.WIDE) costs an
// eighth of one DFMA and carries 64 significant bits instead of 53.  The
// functions here take a double apart into a 64-bit significand and an
// exponent, work in 64-bit fixed point, and round once at the end:
//   rcp_m       1/m by one third-order (Halley-type) step from the hardware's
//               single-precision reciprocal: r (1 + e + e^2), e = 1 - m r;
//   rsqrt_m     m^(-1/2): y (1 + e/2 + 3 e^2/8), e = 1 - m y^2;
//   exp2_neg    2^-f: f = j/1024 + g, a table of 2^(-j/1024) and the Taylor
//               polynomial of 2^-g to g^4 (its last coefficient moved by the
//               fifth term's mean);
//   log2_m      log2 m: m = F (1 + r), F = 1 + j/256, tables of 1/F and
//               log2 F, ln(1 + r) by its Taylor polynomial to r^7
// (table-driven exponential and logarithm in the manner of P. T. P. Tang, ACM
// TOMS 15 (1989) 144 and 16 (1990) 378).  Every intermediate is unsigned: the
// seeds are taken below the true value, so that residuals are positive.
// Errors against 60-digit references before the final rounding: rcp 2^-61.5,
// rsqrt 2^-60, relative; exp2 2^-60.4, log2 2^-60.7, absolute.  (Rounded: see
// pr_math64.cuh.)
//
// Measured rates (per clock and SM): wide 32 x 32-bit multiply-adds 28, 64-bit
// high products 7.5, DFMA 1.7-2.  A division (~45 instructions, 5 wide
// products) takes ~20 cycles of issue per warp and SM against ~8 FP64
// operations of 16 cycles, an exponential ~25 against 11-15 of them.  FP64
// properties of 2.1 M cells of the flame field, divisions, roots,
// exponentials and logarithms moved: 3718 -> 2718 us (954 -> 608 FP64-pipe
// instructions per cell), FP64 inversion 1845 -> 1643 us, FP32 inversion (its
// step in double) of 4.5 M cells 703 -> 535 us.
#pragma once

#include <stdint.h>
#include <string.h>

#ifndef __CUDACC__
#include <math.h>
#ifndef HOST_RCP
#define HOST_RCP(x) (1.0f / (x))
#define HOST_RSQRT(x) (1.0f / sqrtf(x))
#endif
#define I64_FN static inline
#define I64_TAB static const
#else
#define I64_FN __device__ __forceinline__
#define I64_TAB __device__ const
#endif

#include "int64_tables.h"

namespace i64 {

// ------------------------------------------------------------ primitives
I64_FN uint32_t lo32(uint64_t a) { return (uint32_t)a; }
I64_FN uint32_t hi32(uint64_t a) { return (uint32_t)(a >> 32); }
I64_FN uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }

// floor(a b / 2^64), low by at most 2 units (the low x low product dropped)
I64_FN uint64_t mulhi(uint64_t a, uint64_t b)
{
    const uint64_t t = wide(hi32(a), lo32(b)), u = wide(lo32(a), hi32(b));
    return wide(hi32(a), hi32(b)) + (t >> 32) + (u >> 32);
}

// the same for a, b <= 2^63 (not both 2^63): the two middle products' sum fits
// 64 bits, so three multiply-adds and no carry
I64_FN uint64_t mulhi63(uint64_t a, uint64_t b)
{
    const uint64_t t = wide(lo32(a), hi32(b)) + wide(hi32(a), lo32(b));
    return wide(hi32(a), hi32(b)) + (t >> 32);
}

// a b / 2^32 for a 32-bit b, low by less than one unit
I64_FN uint64_t mul32(uint64_t a, uint32_t b) { return wide(hi32(a), b) + (wide(lo32(a), b) >> 32); }

I64_FN uint32_t mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(wide(a, b) >> 32); }

I64_FN uint64_t bits(double x)
{
#ifdef __CUDACC__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
#endif
}
I64_FN double from_bits(uint64_t b)
{
#ifdef __CUDACC__
    return __longlong_as_double((long long)b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}
I64_FN float float_bits(uint32_t b)
{
#ifdef __CUDACC__
    return __uint_as_float(b);
#else
    float x;
    memcpy(&x, &b, 4);
    return x;
#endif
}
I64_FN uint32_t bits_of(float f)
{
#ifdef __CUDACC__
    return __float_as_uint(f);
#else
    uint32_t b;
    memcpy(&b, &f, 4);
    return b;
#endif
}
I64_FN float approx_rcp(float x)
{
#ifdef __CUDACC__
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return HOST_RCP(x);
#endif
}
I64_FN float approx_rsqrt(float x)
{
#ifdef __CUDACC__
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return HOST_RSQRT(x);
#endif
}

// 32-bit operations: a >> s (0 from s = 32 on), the high word of a << s for s
// < 32, leading zeros of a nonzero a, a as a float to nearest
I64_FN uint32_t shr32(uint32_t a, uint32_t s)
{
#ifdef __CUDACC__
    return __funnelshift_rc(a, 0u, s);
#else
    return s < 32 ? a >> s : 0;
#endif
}
I64_FN uint32_t shl_hi32(uint64_t a, uint32_t s)
{
#ifdef __CUDACC__
    return __funnelshift_l(lo32(a), hi32(a), s);
#else
    return hi32(a << s);
#endif
}
I64_FN uint32_t clz32(uint32_t a)
{
#ifdef __CUDACC__
    return (uint32_t)__clz((int)a);
#else
    return (uint32_t)__builtin_clz(a);
#endif
}
I64_FN float to_float(uint32_t a)
{
#ifdef __CUDACC__
    return __uint2float_rn(a);
#else
    return (float)a;
#endif
}

// biased exponent field; significand of a normal number, its leading 1 at bit 63
I64_FN uint32_t expo(uint64_t b) { return (uint32_t)(b >> 52) & 0x7FFu; }
I64_FN uint64_t signif(uint64_t b) { return (b << 11) | 0x8000000000000000ull; }

// m 2^(e - 63) for a normalised m (bit 63 set) and -1022 <= e <= 1022, to nearest
I64_FN uint64_t pack_bits(uint64_t m, int e)
{
    const uint64_t q = (m >> 11) + ((m >> 10) & 1u);
    return q + ((uint64_t)(uint32_t)(1022 + e) << 52);
}

// ------------------------------------------------------------- reciprocal
// 2^64 / m for m = M / 2^63 in [1, 2): in (2^63, 2^64].  The seed is at least
// 2^-24 and at most 5 x 2^-23 (relative) below 1/m: the argument is rounded
// up, three units taken off for the hardware's error of 2^-23.
I64_FN uint64_t rcp_m(uint64_t M)
{
    const float f = float_bits(0x3F800001u + ((uint32_t)(M >> 40) & 0x7FFFFFu));   // (1, 2]
    uint32_t rb = bits_of(approx_rcp(f));
    rb = rb < 0x3F7FFFFFu ? rb : 0x3F7FFFFFu;   // the seed's exponent that of [1/2, 1)
    rb = rb > 0x3F000000u ? rb : 0x3F000000u;
    const uint32_t r0 = ((rb << 8) | 0x80000000u) - 0x300u;   // units 2^-32
    const uint64_t e = 0x8000000000000000ull - mul32(M, r0);   // 1 - m r0, units 2^-63, below 2^43
    const uint32_t s = (uint32_t)(e >> 11);
    const uint64_t t = e + (wide(s, s) >> 41);
    return ((uint64_t)r0 << 32) + (wide(r0, lo32(t)) >> 31) + (wide(r0, hi32(t)) << 1);
}

// ------------------------------------------------------- inverse square root
// x = X / 2^64 in [1/4, 1): x^(-1/2) in (1, 2], units 2^-63
I64_FN uint64_t rsqrt_m(uint64_t X)
{
    // x rounded up to 23 bits as a float, from its bits: [1/2, 1) or [1/4, 1/2)
    const bool small = !(X >> 63);
    const uint64_t Xn = small ? X << 1 : X;
    const float f = float_bits((small ? 0x3E800001u : 0x3F000001u) + ((uint32_t)(Xn >> 40) & 0x7FFFFFu));
    uint32_t yb = bits_of(approx_rsqrt(f));
    yb = yb < 0x3FFFFFFFu ? yb : 0x3FFFFFFFu;
    yb = yb > 0x3F800000u ? yb : 0x3F800000u;
    const uint32_t y0 = ((yb << 8) | 0x80000000u) - 0x400u;   // units 2^-31
    const uint64_t e = 0x4000000000000000ull - mulhi(X, wide(y0, y0));   // 1 - x y0^2, units 2^-62, below 2^44
    const uint32_t s = (uint32_t)(e >> 12);
    const uint64_t t = e + 3u * (wide(s, s) >> 40);
    return ((uint64_t)y0 << 32) + (wide(y0, lo32(t)) >> 31) + (wide(y0, hi32(t)) << 1);
}

// ------------------------------------------------------------------- exp2
// 2^-f for f = F / 2^64 in [0, 1): in (2^62, 2^63], units 2^-63
// (tab: kI64Exp2 or a copy of it in shared memory)
I64_FN uint64_t exp2_neg(uint64_t F, const uint64_t *tab = kI64Exp2)
{
    const uint64_t tj = tab[(uint32_t)(F >> 54)];
    const uint64_t g = (F << 9) & 0x7FFFFFFFFFFFFFFFull;   // g 2^10, units 2^-63
    const uint32_t gh = hi32(g);
    const uint32_t r3 = kI64ExpC3 - mulhi32(gh, kI64ExpC4);   // units 2^-66
    const uint64_t r2 = kI64ExpC2 - mulhi32(gh, r3);          // units 2^-65
    const uint64_t r1 = kI64ExpC1 - mulhi63(g, r2);           // units 2^-64
    return tj - 2 * mulhi63(tj, mulhi63(g, r1));
}

// ------------------------------------------------------------------- log2
// log2 m for m = M / 2^63 in [1, 2): in [0, 1), units 2^-64
I64_FN uint64_t log2_m(uint64_t M)
{
    const uint32_t j = (uint32_t)(M >> 55) & 0xFFu;
    const uint64_t Q = j ? mulhi(M, kI64InvF[j]) : M;
    const uint64_t g = (Q - 0x8000000000000000ull) << 8;   // (m / F - 1) 2^8, units 2^-63
    const uint32_t gh = hi32(g);
    const uint32_t q6 = kI64LogC6 - mulhi32(gh, kI64LogC7);   // units 2^-70
    const uint32_t q5 = kI64LogC5 - mulhi32(gh, q6);
    const uint64_t q4 = kI64LogC4 - mulhi32(gh, q5);          // units 2^-68, up to 35 bits
    const uint64_t q3 = kI64LogC3 - mulhi63(g, q4);
    const uint64_t q2 = kI64LogC2 - mulhi63(g, q3);
    const uint64_t q1 = kI64LogC1 - mulhi63(g, q2);           // units 2^-65
    return kI64Log2F[j] + mulhi63(g, q1);
}

}  // namespace i64
