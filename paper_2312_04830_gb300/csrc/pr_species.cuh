// Per-cell arithmetic of the per-species outputs (Sec. 4.1's species
// networks: standard-state enthalpies and mixture-averaged diffusion with a
// high-pressure correction, Sec. 2), shared by pr_species_props and the
// surrogate's FP64 fallback for its per-species outputs.
//
//   D_km = (sum_{j != k} Y_j / sum_j Y_j) / sum_{j != k} X_j / D_kj, the
//   Chapman-Enskog D_kj = c_kj T^(3/2) / (p Omega_D(T / eps_kj)) from the pair
//   table (1/eps, eps^B, 1/c), times the correction f(T_r, p_r) at the mixture's
//   Kay's-rule state; a species alone in its cell gets D_kk.
#pragma once

#include "pr_device.cuh"

namespace prs {

using prk::M;

// Neufeld et al. (1972) fit of the Lennard-Jones Omega^(1,1)*.
constexpr double kNA = 1.06036, kNB = 0.15610, kNC = 0.19300, kND = 0.47635;
constexpr double kNE = 1.03587, kNF = 1.52996, kNG = 1.76474, kNH = 3.89411;

// Flat per-context table: tc[NS], pc[NS], ie[NS*NS], epsB[NS*NS], ic[NS*NS].
inline size_t dtab_len(int NS) { return 2 * (size_t)NS + 3 * (size_t)NS * NS; }

// Omega_D at T* = Ts, with pw = T*^-B given.  In FP64 this is the general
// form, out of line (36 copies of it would fill the instruction cache); the
// usual temperatures take the fixed-point form below.
template <typename Real>
__device__ __forceinline__ Real omega_d_inline(Real Ts, Real pw)
{
    Real om = Real(kNA) * pw;
    if (Ts < Real(40.0 / kND)) om = M<Real>::fma(Real(kNC), M<Real>::exp(Real(-kND) * Ts), om);
    if (Ts < Real(40.0 / kNF)) om = M<Real>::fma(Real(kNE), M<Real>::exp(Real(-kNF) * Ts), om);
    if (Ts < Real(40.0 / kNH)) om = M<Real>::fma(Real(kNG), M<Real>::exp(Real(-kNH) * Ts), om);
    return om;
}

static __device__ __noinline__ double omega_d_f64(double Ts, double pw) { return omega_d_inline<double>(Ts, pw); }

template <typename Real>
__device__ __forceinline__ Real omega_d(Real Ts, Real pw)
{
    if constexpr (sizeof(Real) == 8)
        return omega_d_f64(Ts, pw);
    else
        return omega_d_inline<Real>(Ts, pw);
}

// ------------------------------------------------ fixed-point pair sums
// For T in [32, 8192) K the pair sums sum_{j != k} n_j / c_kj Omega_kj take
// Omega_D from the integer pipe (pr_int64.cuh).  T is exact in units of
// 2^-51 K; each exponential's argument T D log2(e) / eps_kj is one 64-bit
// product, in units of 2^-53, with log2 of its factor (C, E, G) and of the
// common 1/2 added, so that a term is 2^-argument; Omega_D / 2 is summed in
// units of 2^-62 and leaves as a double after the product with 1 / c_kj.
// Truncations add up to at most 3 x 2^-53 of an argument (0.25 of the sum's
// rounding at the largest share the exponentials take of Omega_D) and
// 2^-60 of the sum.  Per Omega_D ~150 integer instructions replace ~45 FP64
// ones, which hold the FP64 pipe 16 cycles each.
// Omega_D depends on a pair through eps_kj alone, so pairs of equal eps (the
// radicals take their parent molecule's critical constants) share one: 21 for
// the 36 pairs of the nine species here.
struct OmegaFix {
    uint64_t a[3];    // D, F, H log2(e) / eps, units 2^-66 (below 1/4)
    uint64_t pw;      // A eps^B / 2, units 2^-63 (below 2)
};
struct PairFix {
    uint64_t icm;     // 1 / c_kj = icm 2^(ice - 63), icm normalised
    int32_t ice;
    uint16_t k, j;
};
constexpr int kPairs9 = 36;

// 1 - log2 of C, E, G in units of 2^-53, plus one unit for the truncations
constexpr uint64_t kOffC = 0x006BF24BFBC86A2Bull, kOffE = 0x001E5F7E967FD2C7ull, kOffG = 0x0005C704F3E28E63ull;

// Omega_D / 2 in units of 2^-62: Tf = T 2^51, TB = T^-B 2^64; tab: kI64Exp2 (a copy).
__device__ __forceinline__ uint64_t omega_fix(const OmegaFix &c, uint64_t Tf, uint64_t TB, const uint64_t *tab)
{
    uint64_t om = i64::mulhi(TB, c.pw) >> 1;
    const uint64_t p0 = i64::mulhi(Tf, c.a[0]) + kOffC;
    const uint64_t p1 = i64::mulhi(Tf, c.a[1]) + kOffE;
    const uint64_t p2 = i64::mulhi(Tf, c.a[2]) + kOffG;
    // a term of 2^-62 or less of the sum's units is dropped
    const uint32_t n0 = i64::hi32(p0) >> 21, n1 = i64::hi32(p1) >> 21, n2 = i64::hi32(p2) >> 21;
    if (n0 < 62) om += i64::exp2_neg(p0 << 11, tab) >> (n0 + 1u);
    if (n1 < 62) om += i64::exp2_neg(p1 << 11, tab) >> (n1 + 1u);
    if (n2 < 62) om += i64::exp2_neg(p2 << 11, tab) >> (n2 + 1u);
    return om;
}

// Omega_D / c_kj
__device__ __forceinline__ double pair_fix(const PairFix &c, uint64_t om)
{
    const uint64_t q = i64::mulhi(om, c.icm);
    const int z = __clzll((long long)q);
    return i64::from_bits(i64::pack_bits(q << z, c.ice + 3 - z));
}

// Whether T lies in the fixed-point range [32, 8192) K
__device__ __forceinline__ bool fix_range(double T) { return (i64::bits(T) >> 52) - 1028u < 8u; }

template <typename Real>
__device__ __forceinline__ Real corr_factor(const Real *__restrict__ c, int cT, int cP, Real x, Real y)
{
    const Real *Tr = c, *pr = c + cT, *f = c + cT + cP;
    x = fmin(fmax(x, Tr[0]), Tr[cT - 1]);
    y = fmin(fmax(y, pr[0]), pr[cP - 1]);
    int i = 0, j = 0;
    while (i < cT - 2 && x > Tr[i + 1]) ++i;
    while (j < cP - 2 && y > pr[j + 1]) ++j;
    const Real tx = (x - Tr[i]) / (Tr[i + 1] - Tr[i]);
    const Real ty = (y - pr[j]) / (pr[j + 1] - pr[j]);
    const Real *r0 = f + i * cP + j, *r1 = r0 + cP;
    const Real g0 = M<Real>::fma(ty, r0[1] - r0[0], r0[0]);
    const Real g1 = M<Real>::fma(ty, r1[1] - r1[0], r1[0]);
    return M<Real>::fma(tx, g1 - g0, g0);
}

// Mixture-averaged D_k [m^2/s] of one valid cell: y its mass fractions
// (ysum their sum), x its mole fractions (normalised), tab the flat pair table,
// corr the correction table (cT = 0: none); omega(q, TmB): Omega_D of pair q =
// k NS + j from T^-B.
template <typename Real, int NS, typename Omega>
__device__ __forceinline__ void diffusion_sums(const Real (&y)[NS], const Real (&x)[NS], Real ysum, Real T, Real p,
                                               int N, const Real *tab, const Real *corr, int cT, int cP, Real (&D)[NS],
                                               Omega omega)
{
    const Real *tc = tab, *pc = tab + NS, *ie = tab + 2 * NS, *epsB = ie + NS * NS, *ic = epsB + NS * NS;
    Real Tpc = 0, ppc = 0;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        Tpc = M<Real>::fma(x[k], tc[k], Tpc);
        ppc = M<Real>::fma(x[k], pc[k], ppc);
    }
    const Real f = (cT > 0) ? corr_factor<Real>(corr, cT, cP, T / Tpc, p / ppc) : Real(1);
    const Real TmB = prk::pow_neg<Real>(T, kNB);   // T^-B
    Real acc[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) acc[k] = 0;
#pragma unroll
    for (int k = 0; k < NS - 1; ++k) {
        if (k >= N - 1) break;
#pragma unroll
        for (int j = k + 1; j < NS; ++j) {
            if (j >= N) break;
            const int q = k * NS + j;
            const Real om = omega(q, TmB);
            const Real w = om * ic[q];
            acc[k] = M<Real>::fma(x[j], w, acc[k]);
            acc[j] = M<Real>::fma(x[k], w, acc[j]);
        }
    }
    const Real scale = M<Real>::div(f * T * M<Real>::sqrt(T), p);   // f T^(3/2) / p
    // sum_{j != k} y_j from prefix and suffix sums
    Real others[NS];
    Real run = 0;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        others[k] = run;
        run += y[k];
    }
    run = 0;
#pragma unroll
    for (int k = NS - 1; k >= 0; --k) {
        others[k] += run;
        run += y[k];
    }
    const Real iys = M<Real>::rcp(ysum);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
        if (k >= N) break;
        if (acc[k] > Real(0)) {
            D[k] = M<Real>::div(others[k] * iys * scale, acc[k]);
        } else {   // alone in the cell: self-diffusion
            const int q = k * NS + k;
            D[k] = M<Real>::div(scale, omega_d<Real>(T * ie[q], TmB * epsB[q]) * ic[q]);
        }
    }
}

template <typename Real, int NS>
__device__ __forceinline__ void diffusion_cell(const Real (&y)[NS], const Real (&x)[NS], Real ysum, Real T, Real p,
                                               int N, const Real *tab, const Real *corr, int cT, int cP, Real (&D)[NS])
{
    const Real *ie = tab + 2 * NS, *epsB = ie + NS * NS;
    diffusion_sums<Real, NS>(y, x, ysum, T, p, N, tab, corr, cT, cP, D,
                             [&](int q, Real TmB) { return omega_d<Real>(T * ie[q], TmB * epsB[q]); });
}

// h_k^0 / (R T) of one species from its NASA-7 enthalpy record e (molar h =
// ((((e4 T + e3) T + e2) T + e1) T + e0) T + e5) and iRT = 1 / (R T).
template <typename Real>
__device__ __forceinline__ Real h_over_RT(const Real *e, Real T, Real iRT)
{
    const Real h = M<Real>::fma(
        M<Real>::fma(M<Real>::fma(M<Real>::fma(M<Real>::fma(e[4], T, e[3]), T, e[2]), T, e[1]), T, e[0]), T, e[5]);
    return h * iRT;
}

}  // namespace prs
