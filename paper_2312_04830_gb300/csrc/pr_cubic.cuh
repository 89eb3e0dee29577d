// The root of the Peng-Robinson cubic where it has a single one above B, with
// little FP64 work: seeds and root count in FP32, Newton's polish with the
// residual in FP64.
#pragma once

#include <math.h>

#include "pr_int64.cuh"

#ifdef __CUDACC__
#define CUBIC_FDIV(a, b) __fdividef(a, b)
#else
#define CUBIC_FDIV(a, b) ((a) / (b))   // host build (tests)
#endif

namespace prk {

// Conversions on the integer pipe (truncating; magnitudes below FP32's normal
// range become 0): for residuals and derivatives, whose last bits do not matter.
I64_FN float float_of(double x)
{
    const uint64_t b = i64::bits(x);
    const uint32_t hi = i64::hi32(b), lo = i64::lo32(b);
    const uint32_t e = (hi >> 20) & 0x7FFu;
    const uint32_t m = ((hi & 0x000FFFFFu) << 3) | (lo >> 29);
    return i64::float_bits((hi & 0x80000000u) | (e > 896u ? ((e - 896u) << 23) | m : 0u));
}
I64_FN double double_of(float x)   // exact for normal x and 0
{
    const uint32_t b = i64::bits_of(x);
    const uint32_t hi = (b & 0x80000000u) | ((b & 0x7F800000u) ? ((b & 0x7FFFFFFFu) >> 3) + 0x38000000u : 0u);
    return i64::from_bits((uint64_t)hi << 32 | (uint64_t)(b << 29));
}

// Newton's polish of a root z > 0, the residual in FP64, the derivative and the
// quotient in FP32.  The derivative's error is 3e-7 of its terms' magnitudes:
// relative to the derivative at most 3e-3 where that is over 1e-4 of them, so
// each step leaves at most 3e-3 of the distance and the limit is the FP64
// residual's alone, 4 x 2^-53 of its terms over the derivative.  False nearer a
// multiple root (the critical point), where the derivative can have the wrong
// sign, and where the steps have not settled at 1e-10 of z.
I64_FN bool cubic_polish_mixed(double &z, double c2, double c1, double c0)
{
    const float c22f = 2.f * float_of(c2), c1f = float_of(c1);
    float dz = 0.f, zf = 0.f;
#ifdef __CUDACC__
#pragma unroll 1
#endif
    for (int it = 0; it < 12; ++it) {
        const double f = fma(fma(z + c2, z, c1), z, c0);
        zf = float_of(z);
        const float d = fmaf(fmaf(3.f, zf, c22f), zf, c1f);
        if (!(fabsf(d) > 1e-4f * fmaf(fmaf(3.f, zf, fabsf(c22f)), zf, fabsf(c1f)))) return false;
        dz = CUBIC_FDIV(float_of(f), d);
        z -= double_of(dz);
        if (fabsf(dz) <= 4.44e-16f * fabsf(zf)) break;
    }
    return fabsf(dz) <= 1e-10f * fabsf(zf);
}

// Whether the cubic Z^3 + c2 Z^2 + c1 Z + c0 certainly has one root above B,
// and that root.
I64_FN bool cubic_single_root(double c2, double c1, double c0, double B, double &Z)
{
    const double c23 = c2 * (1.0 / 3.0);
    const double P = fma(-c2, c23, c1), Q = fma(c23, fma(2.0 * c23, c23, -c1), c0);
    const float Pf = float_of(P), Qf = float_of(Q), c23f = float_of(c23);
    const float hq = 0.5f * Qf, tp = Pf * (1.f / 3.f), t3 = tp * tp * tp, h2 = hq * hq, disc = h2 + t3;
    const float Bcut = float_of(B) * (1.f - 1e-3f);
    float seed = 0.f;
    bool one = false;   // exactly one seed above B
    if (fabsf(disc) > 1e-4f * (h2 + fabsf(t3))) {   // the sign of the discriminant is settled
        if (disc > 0.f) {
            const float u = cbrtf(-hq - copysignf(sqrtf(disc), hq));
            seed = ((u != 0.f) ? (u - Pf / (3.f * u)) : 0.f) - c23f;
            one = seed > Bcut;
        } else {
            const float m = 2.f * sqrtf(fmaxf(-tp, 0.f));
            float arg = (m > 0.f) ? (3.f * Qf) / (Pf * m) : 0.f;
            arg = fminf(1.f, fmaxf(-1.f, arg));
            const float th = acosf(arg) * (1.f / 3.f);
            seed = m * cosf(th) - c23f;   // the largest; the middle one below B settles the smallest
            one = seed > Bcut && !(m * cosf(th + 4.18879020478639f) - c23f > Bcut);
        }
    }
    if (!one) return false;
    Z = double_of(seed);
    return cubic_polish_mixed(Z, c2, c1, c0) && Z > B;
}

}  // namespace prk
