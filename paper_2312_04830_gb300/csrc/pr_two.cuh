// Numbers as unevaluated sums of two floats, h = the sum rounded.
#pragma once

#ifdef __CUDACC__
#define TWO_FN __device__ __forceinline__
#define TWO_ADD(a, b) __fadd_rn(a, b)
#define TWO_SUB(a, b) __fsub_rn(a, b)
#define TWO_MUL(a, b) __fmul_rn(a, b)
#define TWO_FMA(a, b, c) __fmaf_rn(a, b, c)
#else
#include <math.h>
#define TWO_FN static inline   // host build (tests)
#define TWO_ADD(a, b) ((a) + (b))
#define TWO_SUB(a, b) ((a) - (b))
#define TWO_MUL(a, b) ((a) * (b))
#define TWO_FMA(a, b, c) fmaf(a, b, c)
#endif

namespace prk {

struct Temp2 {
    float h, l;
};
TWO_FN Temp2 temp2_add(Temp2 a, float b)
{
    // two-sum of h and b (Knuth), the tail added and the result renormalised
    const float s = TWO_ADD(a.h, b), bb = TWO_SUB(s, a.h);
    const float e = TWO_ADD(TWO_ADD(TWO_SUB(a.h, TWO_SUB(s, bb)), TWO_SUB(b, bb)), a.l);
    const float h = TWO_ADD(s, e);
    return {h, TWO_SUB(e, TWO_SUB(h, s))};
}
TWO_FN bool temp2_less(Temp2 a, Temp2 b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }

// Whether a b < c d, the products exact (without underflow; false for NaN)
TWO_FN bool product_less(float a, float b, float c, float d)
{
    const float p = TWO_MUL(a, b), q = TWO_MUL(c, d);
    return temp2_less({p, TWO_FMA(a, b, -p)}, {q, TWO_FMA(c, d, -q)});
}

}  // namespace prk
