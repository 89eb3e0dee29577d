// The FP32 composition of a cell for the FP64 inversion's warm start, of up to
// 9 species: mole fractions, mean molar mass and b_m from the FP64 mass
// fractions in 32-bit fixed point, a few 2^-32 of rounding before the one to
// FP32.  From mass fractions rounded to FP32 first, the FP32 root lies farther
// off, and with it the accepted step's result: mean error of T on 1 Mi
// scattered cells 3.81e-14, here 3.61e-14, as from an FP64 composition.  That
// one takes 750 us for 2.1 M cells of the flame field, the 62-bit one of
// pr_fix9.cuh 735, this one 685 (mass fractions rounded first: 676; the second
// launch has since become 50 us shorter).
#pragma once

#include <math.h>

#include "pr_int64.cuh"

namespace prk {

struct WarmTab {
    uint32_t iW[9], b[9];   // 1/W_k, b_k in units of a power of two each
    float sW, sb;           // those of the mean molar mass and of b_m below
};

// From 1/W_k [mol/kg] and b_k [m^3/mol], positive; false where a unit leaves
// FP32's range.
inline bool fill_warm(WarmTab &t, const long double *iW, const long double *b, int N)
{
    long double top_W = 0, top_b = 0;
    for (int k = 0; k < N; ++k) {
        top_W = fmaxl(top_W, iW[k]);
        top_b = fmaxl(top_b, b[k]);
    }
    int eW, eB;   // every 1/W_k below 2^eW, every b_k below 2^eB
    frexpl(top_W, &eW);
    frexpl(top_b, &eB);
    if (eW < -60 || eW > 60 || eB < -60 || eB > 60) return false;
    auto u32 = [](long double v) { return v < 4294967295.0L ? (uint32_t)roundl(v) : 0xFFFFFFFFu; };
    for (int k = 0; k < 9; ++k) {
        t.iW[k] = k < N ? u32(ldexpl(iW[k], 32 - eW)) : 0u;
        t.b[k] = k < N ? u32(ldexpl(b[k], 32 - eB)) : 0u;
    }
    // with s and r of warm_comp, sum y/W = s 2^(eW - 63) and 1/s = r 2^(z - 95);
    // b_m = sum (x 2^31) (b 2^(32 - eB)) 2^(eB - 63)
    t.sW = ldexpf(1.f, -32 - eW);
    t.sb = ldexpf(1.f, eB - 31);
    return true;
}

// Any bits in, mass fractions that the FP64 evaluation refuses among them.
// C: a Comp<float, 9>.
template <class C>
I64_FN void warm_comp(const WarmTab &t, const double (&y)[9], C &c)
{
    uint64_t n[9], s = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < 9; ++k) {
        const uint64_t b = i64::bits(y[k]);
        const uint32_t f = i64::shr32(i64::hi32(i64::signif(b)), 1023u - i64::expo(b));   // y 2^31
        n[k] = i64::wide(f, t.iW[k]);
        s += n[k];
    }
    const uint32_t z = i64::clz32(i64::hi32(s) | 1u);
    const uint32_t r = i64::hi32(i64::rcp_m((s << z) | 0x8000000000000000ull));   // 2^95 / (s 2^z)
    // half a unit of the product, and of what n 2^z loses: truncated, the sum
    // of nine would be 4e-9 short
    const uint64_t half = 0x80000000ull + (r >> 1);
    uint64_t bm = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int k = 0; k < 9; ++k) {
        const uint32_t x = i64::hi32(i64::wide(i64::shl_hi32(n[k], z), r) + half);   // units 2^-31
        bm += i64::wide(x, t.b[k]);
        c.x[k] = i64::to_float(x) * 4.656612873077393e-10f;
    }
    c.Wbar = i64::to_float(r) * (i64::float_bits((127u + z) << 23) * t.sW);
    c.bm = i64::to_float(i64::hi32(bm)) * t.sb;
}

}  // namespace prk
