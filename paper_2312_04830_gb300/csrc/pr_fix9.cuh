// The FP64 evaluation of a cell for up to 9 species with its species sums in
// fixed point on the integer pipe.
//
// The FP64 pipe (2 operations per clock per SM) holds the FP64 property path;
// about 320 of its operations per cell were sums of mole fractions times
// table constants.  Here a mole fraction is a 62-bit fixed-point number in two
// 31-bit limbs, a table constant a 58-bit one in units of a power of two of
// its own sum, and a product adds three 32 x 32-bit multiply-adds into two
// 64-bit accumulators (high x high, and the two middle products; low x low,
// below the sum's last unit, is dropped):
//     3 cycles of the SM's wide-multiply pipe against a DFMA's 16.
// A sum carries 2^-58 of its largest constant and becomes a double once.
//
// With u_k = 1 + kappa_k (1 - sqrt(T / Tc,k)), g_k = sqrt(a_c,k) and
// s_k = sgn(u_k), the van der Waals sums need two of them only,
//     U0 = sum x_k s_k g_k (1 + kappa_k),  U1 = sum x_k s_k g_k kappa_k / sqrt(Tc,k):
//     sqrt(a_m) = S0 = U0 - sqrt(T) U1,  T da_m/dT - a_m = -S0 U0.
//
// Range: T in [32, 4096) K (the NASA-7 polynomials run in T/1024 below the
// switch temperature and T/4096 above it), k_ij = 0, one switch temperature
// in (32, 1024] for all species; other cells and contexts take the general
// form (pr_device.cuh).
#pragma once

#include "pr_cubic.cuh"
#include "pr_kernels.cuh"
#include "pr_warm.cuh"

namespace prk {

struct Mac31 {
    int32_t h, l;   // (h 2^31 + l) units, 0 <= l < 2^31, |value| < 2^58
};

// table constants of one species; the units' exponents are in Fix9
struct Fix9Rec {
    uint64_t iW;                // (1/W) / max(1/W), units 2^-64 (saturated at 1)
    uint64_t T0;                // bits of the temperature where u_k changes sign (beyond: u_k < 0)
    Mac31 b, u0, u1;            // b_k, g_k (1 + kappa_k), g_k kappa_k / sqrt(Tc,k)
    Mac31 nasa[2][6];           // R a_j x (1024 or 4096)^(j-1), j = 1..5; R a_6
};
struct Fix9 {
    Fix9Rec sp[9];
    WarmTab warm;
    int32_t eb, eu0, eu1, en[2], ea6;   // a sum's unit is 2^e
    double iWmax;               // max(1/W) [mol/kg]
    double rWmax;               // its inverse
    uint64_t Tmid;              // bits of the switch temperature
};

struct Fix9Comp {
    int32_t xh[9], xl[9];       // x_k = (xh 2^31 + xl) 2^-62
    double Wbar, iW;            // mean molar mass [kg/mol] and its inverse
};

struct Acc31 {
    int64_t hi, mid;
};
__device__ __forceinline__ void mac(Acc31 &a, int32_t xh, int32_t xl, const Mac31 &c)
{
    a.hi += (int64_t)xh * c.h;
    a.mid += (int64_t)xh * c.l;
    a.mid += (int64_t)xl * c.h;
}
__device__ __forceinline__ int64_t fold(const Acc31 &a) { return a.hi + (a.mid >> 31); }

// v 2^e as a double (rounded once)
__device__ __forceinline__ double fix_to_double(int64_t v, int e)
{
    const bool neg = v < 0;
    const uint64_t m = neg ? 0 - (uint64_t)v : (uint64_t)v;
    const int z = __clzll((long long)m);
    const uint64_t b = i64::pack_bits(m << (z & 63), 63 - z + e) | (neg ? 0x8000000000000000ull : 0);
    return i64::from_bits(m ? b : 0);
}

// a t / 2^62 for a signed a and 0 <= t < 2^62 in limbs
__device__ __forceinline__ int64_t mul62(int64_t a, int32_t th, int32_t tl)
{
    const int32_t ah = (int32_t)(a >> 31), al = (int32_t)(a & 0x7FFFFFFF);
    const int64_t t = (int64_t)ah * tl + (int64_t)al * th;
    return (int64_t)ah * th + (t >> 31);
}

enum Fix9Status : int { kFixOk = 0, kFixBad = 1, kFixGeneral = 2 };

// Mole fractions of a cell.  kFixBad: load_comp would refuse it; kFixGeneral:
// the decision lies within rounding of the limit |sum Y - 1| = 1e-6, which
// load_comp's own order of summation then takes.
__device__ __forceinline__ int fix9_comp(const Fix9 &t, const double (&y)[9], Fix9Comp &c)
{
    uint64_t n[9], s = 0, ys = 0;
    uint32_t carry = 0;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const uint64_t b = i64::bits(y[k]);
        const uint32_t e = (uint32_t)(b >> 52);
        ok = ok && (e < 1024u || b == 0x8000000000000000ull);   // y in [0, 2), or -0
        const uint32_t sh = 1023u - (e & 0x7FFu);
        const uint64_t f = (sh < 64u && e < 2048u) ? i64::signif(b) >> sh : 0;   // y 2^63 (subnormal y: 0)
        ys += f;
        carry += ys < f;
        n[k] = i64::mulhi(f, t.sp[k].iW);
        s += n[k];
    }
    // |sum Y - 1| against 1e-6, in units of 2^-63
    const uint64_t one = 0x8000000000000000ull;
    const uint64_t d = ys > one ? ys - one : one - ys;
    constexpr uint64_t lim = 9223372036855ull;   // 1e-6 x 2^63
    if (!ok || carry || d > lim + 0x100000ull) return kFixBad;
    if (d > lim - 0x100000ull) return kFixGeneral;   // within 1e-13 of the limit
    const int z = __clzll((long long)s);
    const uint64_t sn = s << z;                     // s > 0: the mass fractions sum to 1
    const uint64_t r = i64::rcp_m(sn);              // 2^64 / (sn / 2^63)
    // r is at most two units high (its residual is rounded up by less than one
    // unit of 2^-63): with two taken off, x of a species alone in its cell
    // stays below 2^63, the end of xh
    const uint64_t rx = r - 2;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const uint64_t x = i64::mulhi(n[k] << z, rx);   // units 2^-63
        c.xh[k] = (int32_t)(x >> 32);
        c.xl[k] = (int32_t)(i64::lo32(x) >> 1);
    }
    // sum y/W = sn 2^-(63 + z) max(1/W)
    c.iW = i64::from_bits(i64::pack_bits(sn, -z)) * t.iWmax;
    c.Wbar = i64::from_bits(i64::pack_bits(r, z - 1)) * t.rWmax;
    return kFixOk;
}

// The physical root, as cubic_phys_roots and select_root: the common case of
// one root above B directly, the others through them.  Returns the status.
__device__ __forceinline__ int cubic_root_fix(double c2, double c1, double c0, double A, double B, double &Z, int &nroots)
{
    if (cubic_single_root(c2, c1, c0, B, Z)) {
        nroots = 1;
        return kOk;
    }
    double zr[3];
    nroots = cubic_phys_roots<double>(c2, c1, c0, B, zr);
    return select_root<double>(zr, nroots, A, B, Z);
}

// T in [32, 4096)
__device__ __forceinline__ bool fix9_range(double T) { return (i64::bits(T) >> 52) - 1028u < 7u; }

// Z, h and the ideal-gas cv of a cell with T in the fixed-point range (as
// thermo<..., CP = false>).
__device__ __forceinline__ void fix9_thermo(const Fix9 &t, const Fix9Comp &c, double T, double p, Thermo<double> &o)
{
    const uint64_t bT = i64::bits(T);
    Acc31 ab = {0, 0}, a0 = {0, 0}, a1 = {0, 0};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        mac(ab, c.xh[k], c.xl[k], t.sp[k].b);
        const bool neg = bT > t.sp[k].T0;
        const int32_t xh = neg ? -c.xh[k] : c.xh[k], xl = neg ? -c.xl[k] : c.xl[k];
        mac(a0, xh, xl, t.sp[k].u0);
        mac(a1, xh, xl, t.sp[k].u1);
    }
    const double bm = fix_to_double(fold(ab), t.eb);
    const double U0 = fix_to_double(fold(a0), t.eu0), U1 = fix_to_double(fold(a1), t.eu1);
    const double sqT = m64::sqrt(T);
    const double S0 = fma(-sqT, U1, U0);
    const double am = S0 * S0;
    const double RT = kR * T;
    const double iRT = m64::rcp(RT);
    const double pRT = p * iRT;
    const double B = bm * pRT, A = am * pRT * iRT;
    const double c2 = B - 1.0, c1 = A - B * fma(3.0, B, 2.0), c0 = B * (B + fma(B, B, -A));
    double Z;
    o.status = cubic_root_fix(c2, c1, c0, A, B, Z, o.nroots);
    if (o.status == kNoRoot) return;
    const double Lr = m64::log1p(m64::div(2.0 * kSqrt2 * B, fma(1.0 - kSqrt2, B, Z)));

    // ideal gas: cp = sum_j A_j tau^j, h = T sum_j A_j tau^j / (j + 1) + A_6
    const bool lowT = bT < t.Tmid;
    int64_t An[5], A6;
    int en;
    auto sums = [&](auto range) {
        constexpr int r = decltype(range)::value;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            Acc31 a = {0, 0};
#pragma unroll
            for (int k = 0; k < 9; ++k) mac(a, c.xh[k], c.xl[k], t.sp[k].nasa[r][j]);
            if (j < 5) An[j] = fold(a);
            else A6 = fold(a);
        }
        en = t.en[r];
    };
    if (lowT) sums(std::integral_constant<int, 0>());
    else sums(std::integral_constant<int, 1>());
    // tau = T / 1024 (T / 4096), units 2^-62
    const uint64_t tau = i64::signif(bT) >> ((lowT ? 1034u : 1036u) - (uint32_t)(bT >> 52));
    const int32_t th = (int32_t)(tau >> 31), tl = (int32_t)(tau & 0x7FFFFFFFu);
    const int64_t cpi = An[0] + mul62(An[1] + mul62(An[2] + mul62(An[3] + mul62(An[4], th, tl), th, tl), th, tl), th, tl);
    constexpr int32_t f3h = 0x2AAAAAAA, f3l = 0x55555555;   // 1/3, 1/5 in units of 2^-62
    constexpr int32_t f5h = 0x19999999, f5l = 0x4CCCCCCD;
    const int64_t hpi =
        An[0] + mul62((An[1] >> 1) + mul62(mul62(An[2], f3h, f3l) +
                                               mul62((An[3] >> 2) + mul62(mul62(An[4], f5h, f5l), th, tl), th, tl),
                                           th, tl), th, tl);
    const double cp_ig = fix_to_double(cpi, en);
    const double h_ig = fma(T, fix_to_double(hpi, en), fix_to_double(A6, t.ea6));

    const double kL = m64::div(Lr, 2.0 * kSqrt2 * bm);
    o.Z = Z;
    o.h = (h_ig + fma(RT, Z - 1.0, -(S0 * U0) * kL)) * c.iW;
    o.cv_ig_molar = cp_ig - kR;
    o.rho_mol = 0;
    o.cp = 0;
    o.dpdT = 0;
    o.dpdV = 0;
}

// launcher and resident CTAs per SM of the inversion kernels (pr_inst_fix9.cu)
// (htab32: the context's HostTab9<float>)
void launch_newton_fix(const NewtonArgs<double> &a, const Fix9 &t, const void *htab32, const int occ[3], int sms,
                       cudaStream_t st);
void occupancy_newton_fix(int occ[3]);

}  // namespace prk
