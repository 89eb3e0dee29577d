// Per-species outputs of the property networks (Sec. 4.1 lists, among the
// seven networks, the nondimensional standard-state enthalpies and the
// mixture-averaged diffusion coefficients of every species; Sec. 2 names the
// binary diffusion model with Takahashi's high-pressure correction):
//
//   h_k^0 / (R T)   NASA-7 fit of species k;
//   D_km            = (1 - Y_k) / sum_{j != k} X_j / D_kj  (mass-fraction form
//                     of the mixture average), 1 - Y_k evaluated as
//                     sum_{j != k} Y_j / sum_j Y_j (no cancellation as Y_k -> 1,
//                     which FP32 inputs reach), a species alone in its cell
//                     taking its self-diffusion coefficient D_kk;
//   D_kj            Chapman-Enskog, D_kj = c_kj T^(3/2) / (p Omega_D(T / eps_kj)),
//                     c_kj = 0.0266 / (M_kj^(1/2) sigma_kj^2) [m^2 Pa/(s K^1.5)]
//                     (0.00266 cm^2 bar units), Neufeld's Omega_D,
//                     sigma = 0.809 Vc^(1/3) [A], eps/k = Tc / 1.2593 (Chung's
//                     corresponding states), sigma_kj arithmetic, eps_kj
//                     geometric, M_kj = 2 / (1/W_k + 1/W_j) [g/mol];
//   f(T_r, p_r)     optional caller table multiplying every D_kj p, bilinear
//                     and edge-clamped, at the mixture's Kay's-rule state.
//
// One thread per cell.  The pair terms are symmetric, so each unordered pair
// evaluates its collision integral once and feeds both species' sums.  In
// Neufeld's Omega_D = A T*^-B + C e^(-D T*) + E e^(-F T*) + G e^(-H T*) the
// power term factors as A T^-B eps_kj^B (one power per cell, a constant per
// pair), and an exponential term whose argument exceeds 40 is dropped: it is
// below 8e-18 while Omega_D >= 0.4, under half an FP64 ulp of the sum.  Pair
// constants (1/eps, eps^B, 1/c) are derived on the host when the context is
// created and staged in shared memory per CTA.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "pr_device.cuh"
#include "pr_internal.h"
#include "pr_species.cuh"

namespace {

using prk::M;
using prk::SpeciesRec;
using prs::corr_factor;
using prs::dtab_len;
using prs::omega_d;

constexpr int kSpBlock = 128;
constexpr int kCorrMax = 64;
constexpr int kCorrFloats = 2 * kCorrMax + kCorrMax * kCorrMax;

template <typename Real>
struct SpArgs {
    int64_t n, ldY, ldo;
    const Real *T, *p, *Y;
    Real *hk, *Dk;
    int32_t *status;
    const SpeciesRec<Real> *sp;
    const Real *dtab;
    const Real *corr;     // Tr[cT], pr[cP], f[cT][cP]; cT = 0: no correction
    int N, cT, cP;
};

template <typename Real, int NS>
__global__ void __launch_bounds__(kSpBlock) species_kernel(const SpArgs<Real> a)
{
    __shared__ Real s_h[2][NS][6];
    __shared__ Real s_tmid[NS], s_iW[NS];
    __shared__ Real s_tab[2 * NS + 3 * NS * NS];
    for (int e = threadIdx.x; e < NS * 6; e += blockDim.x) {
        const int k = e / 6, j = e % 6;
        s_h[0][k][j] = a.sp[k].h_lo[j];
        s_h[1][k][j] = a.sp[k].h_hi[j];
    }
    for (int k = threadIdx.x; k < NS; k += blockDim.x) {
        s_tmid[k] = a.sp[k].T_mid;
        s_iW[k] = a.sp[k].inv_W;
    }
    for (int e = threadIdx.x; e < 2 * NS + 3 * NS * NS; e += blockDim.x) s_tab[e] = a.dtab[e];
    __syncthreads();

    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
        const Real T = __ldg(a.T + i), p = __ldg(a.p + i);
        Real y[NS], x[NS];
        Real ysum = 0, s = 0;
        bool ok = (T > Real(0)) && (p > Real(0)) && M<Real>::finite(T) && M<Real>::finite(p);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            y[k] = (k < a.N) ? __ldg(a.Y + (int64_t)k * a.ldY + i) : Real(0);
            ok = ok && (y[k] >= Real(0)) && M<Real>::finite(y[k]);
            ysum += y[k];
            x[k] = y[k] * s_iW[k];
            s += x[k];
        }
        ok = ok && (M<Real>::fabs(ysum - Real(1)) <= Real(1e-6)) && (s > Real(0));
        if (a.status) a.status[i] = ok ? prk::kOk : prk::kBadInput;
        if (!ok) {
            const Real nanv = M<Real>::nan();
            for (int k = 0; k < a.N; ++k) {
                if (a.hk) a.hk[(int64_t)k * a.ldo + i] = nanv;
                if (a.Dk) a.Dk[(int64_t)k * a.ldo + i] = nanv;
            }
            continue;
        }
        if (a.hk) {
            const Real iRT = M<Real>::rcp(Real(prk::kR) * T);
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (k >= a.N) break;
                a.hk[(int64_t)k * a.ldo + i] = prs::h_over_RT<Real>(s_h[T < s_tmid[k] ? 0 : 1][k], T, iRT);
            }
        }
        if (a.Dk) {
            const Real inv_s = M<Real>::rcp(s);
#pragma unroll
            for (int k = 0; k < NS; ++k) x[k] *= inv_s;
            Real D[NS];
            prs::diffusion_cell<Real, NS>(y, x, ysum, T, p, a.N, s_tab, a.corr, a.cT, a.cP, D);
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                if (k >= a.N) break;
                a.Dk[(int64_t)k * a.ldo + i] = D[k];
            }
        }
    }
}

// The FP32 outputs of up to 9 species.  Omega_D depends on a pair through
// eps_kj alone, so the distinct eps (21 of the 36 pairs' for the nine species
// here: the radicals take their parent molecule's critical constants) are
// evaluated first, into shared memory, and the pair sums read them from there:
// the same operations on the same numbers, in 1800 instructions per cell in
// place of 2610 (the kernel is issue-bound).
struct SpShare9 {
    float ie[36], epsB[36];   // of each distinct eps
    int32_t n;
    int32_t of[81];           // pair k 9 + j: its distinct eps
};

__global__ void __launch_bounds__(kSpBlock) species_share_kernel(const __grid_constant__ SpArgs<float> a,
                                                                 const __grid_constant__ SpShare9 t)
{
    __shared__ float s_h[2][9][6];
    __shared__ float s_tmid[9], s_iW[9];
    __shared__ float s_tab[2 * 9 + 3 * 81];
    __shared__ float s_om[36][kSpBlock];   // this thread's column: no barrier between uses
    for (int e = threadIdx.x; e < 9 * 6; e += blockDim.x) {
        const int k = e / 6, j = e % 6;
        s_h[0][k][j] = a.sp[k].h_lo[j];
        s_h[1][k][j] = a.sp[k].h_hi[j];
    }
    for (int k = threadIdx.x; k < 9; k += blockDim.x) {
        s_tmid[k] = a.sp[k].T_mid;
        s_iW[k] = a.sp[k].inv_W;
    }
    for (int e = threadIdx.x; e < 2 * 9 + 3 * 81; e += blockDim.x) s_tab[e] = a.dtab[e];
    __syncthreads();
    const int tid = threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + tid; i < a.n; i += stride) {
        const float T = __ldg(a.T + i), p = __ldg(a.p + i);
        float y[9], x[9];
        float ysum = 0, s = 0;
        bool ok = (T > 0.f) && (p > 0.f) && M<float>::finite(T) && M<float>::finite(p);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            y[k] = (k < a.N) ? __ldg(a.Y + (int64_t)k * a.ldY + i) : 0.f;
            ok = ok && (y[k] >= 0.f) && M<float>::finite(y[k]);
            ysum += y[k];
            x[k] = y[k] * s_iW[k];
            s += x[k];
        }
        ok = ok && (M<float>::fabs(ysum - 1.f) <= 1e-6f) && (s > 0.f);
        if (a.status) a.status[i] = ok ? prk::kOk : prk::kBadInput;
        if (!ok) {
            const float nanv = M<float>::nan();
            for (int k = 0; k < a.N; ++k) {
                if (a.hk) a.hk[(int64_t)k * a.ldo + i] = nanv;
                if (a.Dk) a.Dk[(int64_t)k * a.ldo + i] = nanv;
            }
            continue;
        }
        if (a.hk) {
            const float iRT = M<float>::rcp(float(prk::kR) * T);
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                if (k >= a.N) break;
                a.hk[(int64_t)k * a.ldo + i] = prs::h_over_RT<float>(s_h[T < s_tmid[k] ? 0 : 1][k], T, iRT);
            }
        }
        if (a.Dk) {
            const float TmB = prk::pow_neg<float>(T, prs::kNB);
#pragma unroll 3
            for (int u = 0; u < t.n; ++u) s_om[u][tid] = prs::omega_d<float>(T * t.ie[u], TmB * t.epsB[u]);
            const float inv_s = M<float>::rcp(s);
#pragma unroll
            for (int k = 0; k < 9; ++k) x[k] *= inv_s;
            float D[9];
            prs::diffusion_sums<float, 9>(y, x, ysum, T, p, a.N, s_tab, a.corr, a.cT, a.cP, D,
                                          [&](int q, float) { return s_om[t.of[q]][tid]; });
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                if (k >= a.N) break;
                a.Dk[(int64_t)k * a.ldo + i] = D[k];
            }
        }
    }
}

// The FP64 outputs of up to 9 species without a correction table: the pair
// sums in fixed point (pr_species.cuh), every table in the kernel's parameter
// space, cells outside the fixed-point range through the general form.
// D_k = (sum_{j != k} y_j / sum_j y_j) f T^1.5 / p / sum_{j != k} x_j / D_kj p / T^1.5
// with moles per kg n_j = y_j / W_j in place of x_j = n_j / sum n (one factor
// per cell); h_k / (R T) = sum_j a_j T^j / (j + 1) + a_6 / T.
struct SpFix9 {
    prs::OmegaFix om[prs::kPairs9];     // of each distinct eps
    prs::PairFix pair[prs::kPairs9];    // ordered by eps
    int32_t first[prs::kPairs9 + 1];    // a distinct eps's first pair
    int32_t n_om;
    double h[2][9][6];        // a_1, a_2/2, ..., a_5/5, a_6 of the low and the high range
    double tmid[9], iW[9];
};

static __device__ __noinline__ void diffusion_general9(const double *y9, const double *x9, double ysum, double T,
                                                       double p, int N, const double *tab, const double *corr, int cT,
                                                       int cP, double *D9)
{
    double y[9], x[9], D[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        y[k] = y9[k];
        x[k] = x9[k];
    }
    prs::diffusion_cell<double, 9>(y, x, ysum, T, p, N, tab, corr, cT, cP, D);
#pragma unroll
    for (int k = 0; k < 9; ++k) D9[k] = D[k];
}

__global__ void __launch_bounds__(kSpBlock, 6) species_fix_kernel(const __grid_constant__ SpArgs<double> a,
                                                               const __grid_constant__ SpFix9 t)
{
    __shared__ uint64_t s_exp2[1024];
    __shared__ double s_x[9][kSpBlock], s_acc[9][kSpBlock];   // this thread's columns: no barrier between uses
    if (a.Dk) {
        for (int e = threadIdx.x; e < 512; e += blockDim.x)
            reinterpret_cast<ulonglong2 *>(s_exp2)[e] = reinterpret_cast<const ulonglong2 *>(kI64Exp2)[e];
        __syncthreads();
    }
    const double nanv = M<double>::nan();
    const int tid = threadIdx.x, N = a.N;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + tid; i < a.n; i += stride) {
        const double T = __ldg(a.T + i), p = __ldg(a.p + i);
        double y[9];
        double ysum = 0, s = 0;
        bool ok = (T > 0.0) && (p > 0.0) && M<double>::finite(T) && M<double>::finite(p);
#pragma unroll
        for (int k = 0; k < 9; ++k) y[k] = (k < N) ? __ldg(a.Y + (int64_t)k * a.ldY + i) : 0.0;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            ok = ok && prk::nonneg_finite(y[k]);
            ysum += y[k];
            const double x = y[k] * t.iW[k];
            s_x[k][tid] = x;
            s_acc[k][tid] = 0.0;
            s += x;
        }
        ok = ok && (M<double>::fabs(ysum - 1.0) <= 1e-6) && (s > 0.0);
        if (a.status) a.status[i] = ok ? prk::kOk : prk::kBadInput;
        if (!ok) {
            for (int k = 0; k < N; ++k) {
                if (a.hk) a.hk[(int64_t)k * a.ldo + i] = nanv;
                if (a.Dk) a.Dk[(int64_t)k * a.ldo + i] = nanv;
            }
            continue;
        }
        if (a.Dk && !prs::fix_range(T)) {
            const double inv_s = M<double>::rcp(s);
            double x[9], D[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) x[k] = s_x[k][tid] * inv_s;
            diffusion_general9(y, x, ysum, T, p, N, a.dtab, a.corr, 0, 0, D);
            for (int k = 0; k < N; ++k) a.Dk[(int64_t)k * a.ldo + i] = D[k];
        } else if (a.Dk) {
            // s T^(3/2) / (p sum_j y_j)
            const double scale = M<double>::div(s * T * M<double>::sqrt(T), p * ysum);
            const uint64_t bT = i64::bits(T);
            const uint64_t Tf = i64::signif(bT) >> (1035u - (uint32_t)(bT >> 52));
            const uint64_t TB = m64::pow_frac_fixed(bT, (uint64_t)(prs::kNB * 18446744073709551616.0));
            // in loops: unrolled, their ~6000 instructions miss the instruction
            // cache (the accumulators then live in shared memory)
#pragma unroll 1
            for (int u = 0; u < t.n_om; ++u) {
                const uint64_t om = prs::omega_fix(t.om[u], Tf, TB, s_exp2);
#pragma unroll 1
                for (int q = t.first[u]; q < t.first[u + 1]; ++q) {
                    const double w = prs::pair_fix(t.pair[q], om);
                    const int k = t.pair[q].k, j = t.pair[q].j;
                    s_acc[k][tid] = fma(s_x[j][tid], w, s_acc[k][tid]);
                    s_acc[j][tid] = fma(s_x[k][tid], w, s_acc[j][tid]);
                }
            }
            // (y read again: held across the pairs it would cost 18 registers)
#pragma unroll
            for (int k = 0; k < 9; ++k) y[k] = (k < N) ? __ldg(a.Y + (int64_t)k * a.ldY + i) : 0.0;
            // sum_{j != k} y_j from prefix and suffix sums
            double others[9];
            double run = 0;
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                others[k] = run;
                run += y[k];
            }
            run = 0;
#pragma unroll
            for (int k = 8; k >= 0; --k) {
                others[k] += run;
                run += y[k];
            }
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                if (k >= N) break;
                const double acc = s_acc[k][tid];
                double D;
                if (acc > 0.0) {
                    D = M<double>::div(others[k] * scale, acc);
                } else {   // alone in the cell: self-diffusion, the general form
                    const double *ie = a.dtab + 18, *epsB = ie + 81, *ic = epsB + 81;
                    const double TmB = prk::pow_neg<double>(T, prs::kNB);
                    D = M<double>::div(M<double>::div(T * M<double>::sqrt(T), p),
                                       prs::omega_d<double>(T * ie[10 * k], TmB * epsB[10 * k]) * ic[10 * k]);
                }
                a.Dk[(int64_t)k * a.ldo + i] = D;
            }
        }
        // (last: hk may lie over Y, which is read again above)
        if (a.hk) {
            const double iT = M<double>::rcp(T);
#pragma unroll 1
            for (int k = 0; k < N; ++k) {
                const bool low = prk::lt_pos(T, t.tmid[k]);
                const double *e = t.h[low ? 0 : 1][k];
                const double h = fma(fma(fma(fma(e[4], T, e[3]), T, e[2]), T, e[1]), T, e[0]);
                a.hk[(int64_t)k * a.ldo + i] = fma(e[5], iT, h);
            }
        }
    }
}

// Bilger's mixture fraction per cell: Z = (sum_k b_k Y_k - beta_ox) / (beta_fuel - beta_ox).
template <typename Real>
__global__ void __launch_bounds__(kSpBlock) bilger_kernel(int64_t n, const Real *__restrict__ Y, int64_t ldY,
                                                          int N, const Real *__restrict__ coef, Real *Z)
{
    const Real bo = coef[N], ir = coef[N + 1];
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        Real beta = 0;
        for (int k = 0; k < N; ++k) beta = M<Real>::fma(__ldg(coef + k), __ldg(Y + (int64_t)k * ldY + i), beta);
        Z[i] = (beta - bo) * ir;
    }
}

template <typename Real, int NS>
void launch_species(const SpArgs<Real> &a, int occ, int sms, cudaStream_t st)
{
    int64_t need = (a.n + kSpBlock - 1) / kSpBlock;
    const int64_t cap = (int64_t)occ * sms;
    const int g = (int)(need < cap ? need : cap);
    species_kernel<Real, NS><<<g, kSpBlock, 0, st>>>(a);
}

template <typename Real, int NS>
int occ_of()
{
    int o = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, species_kernel<Real, NS>, kSpBlock, 0);
    return o > 0 ? o : 1;
}

}  // namespace

namespace prgb {

// The fixed-point kernel's tables; false where a pair constant leaves its
// range (eps_kj below 22.5 K, or a collision integral above 4 at 32 K).
static bool fill_fix9(SpFix9 &f, const pr_species_table *tbl)
{
    typedef long double ld;   // at least 64 significant bits on x86-64 and aarch64
    const int N = tbl->n_species;
    std::memset(&f, 0, sizeof(f));
    const ld log2e = 1.442695040888963407359924681001892137L;
    const ld D[3] = {(ld)prs::kND, (ld)prs::kNF, (ld)prs::kNH};
    for (int k = 0; k < N; ++k) {
        f.tmid[k] = tbl->T_mid[k];
        f.iW[k] = 1.0 / (tbl->W[k] * 1e-3);
        for (int j = 0; j < 6; ++j) {
            f.h[0][k][j] = j < 5 ? tbl->nasa_lo[7 * k + j] / (j + 1) : tbl->nasa_lo[7 * k + 5];
            f.h[1][k][j] = j < 5 ? tbl->nasa_hi[7 * k + j] / (j + 1) : tbl->nasa_hi[7 * k + 5];
        }
    }
    // the distinct eps_kj^2 ~ Tc_k Tc_j, in order of first appearance, and their pairs
    int n_pair = 0;
    bool seen[9][9] = {};
    for (int k0 = 0; k0 < N; ++k0)
        for (int j0 = k0 + 1; j0 < N; ++j0) {
            if (seen[k0][j0]) continue;
            const ld e2 = (ld)tbl->Tc[k0] * (ld)tbl->Tc[j0], eps = sqrtl(e2) / 1.2593L;
            const ld pw = 0.5L * (ld)prs::kNA * powl(eps, (ld)prs::kNB);
            // Omega_D / 2 at 32 K, its largest, within the sum's four units (and A eps^B / 2 below 2)
            if (!(eps > 22.5L) || !(pw < 2.0L) || !(pw * powl(32.0L, -(ld)prs::kNB) < 2.4L)) return false;
            prs::OmegaFix &o = f.om[f.n_om];
            for (int m = 0; m < 3; ++m) o.a[m] = (uint64_t)roundl(ldexpl(D[m] * log2e / eps, 66));
            o.pw = (uint64_t)roundl(ldexpl(pw, 63));
            f.first[f.n_om++] = n_pair;
            for (int k = k0; k < N; ++k)
                for (int j = k + 1; j < N; ++j) {
                    if (seen[k][j] || (ld)tbl->Tc[k] * (ld)tbl->Tc[j] != e2) continue;
                    seen[k][j] = true;
                    const ld sig = 0.5L * 0.809L * (cbrtl((ld)tbl->Vc[k]) + cbrtl((ld)tbl->Vc[j]));
                    const ld Mkj = 2.0L / (1.0L / (ld)tbl->W[k] + 1.0L / (ld)tbl->W[j]);
                    int e;
                    const ld fr = frexpl(sqrtl(Mkj) * sig * sig / 0.0266L, &e);   // 1 / c_kj = fr 2^e, fr in [1/2, 1)
                    const ld m64 = roundl(ldexpl(fr, 64));
                    if (!(m64 < 18446744073709551616.0L) || e < -900 || e > 900) return false;
                    f.pair[n_pair].icm = (uint64_t)m64;
                    f.pair[n_pair].ice = e - 1;
                    f.pair[n_pair].k = (uint16_t)k;
                    f.pair[n_pair].j = (uint16_t)j;
                    ++n_pair;
                }
        }
    f.first[f.n_om] = n_pair;
    return true;
}

// Pair constants from the validated species table (entries of species >= N
// are zero and never read).
pr_status species_tables_init(pr_ctx *c, const pr_species_table *tbl)
{
    const int N = tbl->n_species, NS = c->ns_pad;
    std::vector<double> t(dtab_len(NS), 0.0);
    double *tc = t.data(), *pc = tc + NS, *ie = pc + NS, *epsB = ie + NS * NS, *ic = epsB + NS * NS;
    for (int k = 0; k < N; ++k) {
        tc[k] = tbl->Tc[k];
        pc[k] = tbl->pc[k];
    }
    for (int k = 0; k < N; ++k)
        for (int j = 0; j < N; ++j) {
            const double sk = 0.809 * std::cbrt(tbl->Vc[k]), sj = 0.809 * std::cbrt(tbl->Vc[j]);
            const double sig = 0.5 * (sk + sj);
            const double eps = std::sqrt((tbl->Tc[k] / 1.2593) * (tbl->Tc[j] / 1.2593));
            const double Mkj = 2.0 / (1.0 / tbl->W[k] + 1.0 / tbl->W[j]);
            const double ckj = 0.0266 / (std::sqrt(Mkj) * sig * sig);
            ie[k * NS + j] = 1.0 / eps;
            epsB[k * NS + j] = std::pow(eps, prs::kNB);
            ic[k * NS + j] = 1.0 / ckj;
        }
    if (NS == 9) {
        SpFix9 *f = new (std::nothrow) SpFix9();
        if (!f) {
            set_error("pr_create: host allocation failed");
            return PR_ENOMEM;
        }
        if (fill_fix9(*f, tbl)) c->h_spfix = f;
        else delete f;
    }
    std::vector<float> t32(t.size());
    for (size_t e = 0; e < t.size(); ++e) t32[e] = (float)t[e];
    PR_CUDA_TRY(cudaMalloc(&c->d_dtab64, t.size() * sizeof(double)));
    PR_CUDA_TRY(cudaMalloc(&c->d_dtab32, t.size() * sizeof(float)));
    PR_CUDA_TRY(cudaMalloc(&c->d_corr64, kCorrFloats * sizeof(double)));
    PR_CUDA_TRY(cudaMalloc(&c->d_corr32, kCorrFloats * sizeof(float)));
    PR_CUDA_TRY(cudaMalloc(&c->d_bilger64, (N + 2) * sizeof(double)));
    PR_CUDA_TRY(cudaMalloc(&c->d_bilger32, (N + 2) * sizeof(float)));
    c->has_bilger = 0;
    PR_CUDA_TRY(cudaMemcpy(c->d_dtab64, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice));
    PR_CUDA_TRY(cudaMemcpy(c->d_dtab32, t32.data(), t32.size() * sizeof(float), cudaMemcpyHostToDevice));
    c->corr_nT = c->corr_nP = 0;
    c->occ_species[0] = (NS == 9) ? occ_of<double, 9>() : occ_of<double, 32>();
    c->occ_spfix = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c->occ_spfix, species_fix_kernel, kSpBlock, 0);
    c->occ_spfix = c->occ_spfix > 0 ? c->occ_spfix : 1;
    if (NS == 9) {
        SpShare9 *sh = new (std::nothrow) SpShare9();
        if (!sh) {
            set_error("pr_create: host allocation failed");
            return PR_ENOMEM;
        }
        c->h_spshare = sh;
        const float *ie32 = t32.data() + 2 * NS, *eb32 = ie32 + NS * NS;
        for (int k = 0; k < N; ++k)
            for (int j = k + 1; j < N; ++j) {
                const int q = k * NS + j;
                int u = 0;
                while (u < sh->n && !(sh->ie[u] == ie32[q] && sh->epsB[u] == eb32[q])) ++u;
                if (u == sh->n) {
                    sh->ie[u] = ie32[q];
                    sh->epsB[u] = eb32[q];
                    ++sh->n;
                }
                sh->of[q] = u;
            }
        c->occ_species[1] = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c->occ_species[1], species_share_kernel, kSpBlock, 0);
        c->occ_species[1] = c->occ_species[1] > 0 ? c->occ_species[1] : 1;
    } else {
        c->occ_species[1] = occ_of<float, 32>();
    }
    return PR_OK;
}

void species_tables_free(pr_ctx *c)
{
    cudaFree(c->d_dtab64);
    cudaFree(c->d_dtab32);
    cudaFree(c->d_corr64);
    cudaFree(c->d_corr32);
    cudaFree(c->d_bilger64);
    cudaFree(c->d_bilger32);
    delete static_cast<SpFix9 *>(c->h_spfix);
    delete static_cast<SpShare9 *>(c->h_spshare);
}

}  // namespace prgb

extern "C" {

pr_status pr_set_diffusion_correction(pr_ctx *ctx, const pr_diffusion_correction *corr)
{
    PR_CHECK_ARG(ctx != nullptr, "pr_set_diffusion_correction: null context");
    if (corr == nullptr) {
        PR_CUDA_TRY(cudaDeviceSynchronize());
        ctx->corr_nT = ctx->corr_nP = 0;
        return PR_OK;
    }
    const int nT = corr->n_Tr, nP = corr->n_pr;
    PR_CHECK_ARG(nT >= 2 && nT <= kCorrMax && nP >= 2 && nP <= kCorrMax,
                 "pr_set_diffusion_correction: table %d x %d outside 2..%d", nT, nP, kCorrMax);
    PR_CHECK_ARG(corr->Tr && corr->pr && corr->f, "pr_set_diffusion_correction: null array");
    for (int i = 0; i < nT; ++i)
        PR_CHECK_ARG(std::isfinite(corr->Tr[i]) && (i == 0 || corr->Tr[i] > corr->Tr[i - 1]),
                     "pr_set_diffusion_correction: Tr must be finite and strictly increasing");
    for (int j = 0; j < nP; ++j)
        PR_CHECK_ARG(std::isfinite(corr->pr[j]) && (j == 0 || corr->pr[j] > corr->pr[j - 1]),
                     "pr_set_diffusion_correction: pr must be finite and strictly increasing");
    for (int e = 0; e < nT * nP; ++e)
        PR_CHECK_ARG(std::isfinite(corr->f[e]) && corr->f[e] >= 0.0,
                     "pr_set_diffusion_correction: factors must be finite and >= 0");
    std::vector<double> t(nT + nP + nT * nP);
    std::memcpy(t.data(), corr->Tr, nT * sizeof(double));
    std::memcpy(t.data() + nT, corr->pr, nP * sizeof(double));
    std::memcpy(t.data() + nT + nP, corr->f, (size_t)nT * nP * sizeof(double));
    std::vector<float> t32(t.size());
    for (size_t e = 0; e < t.size(); ++e) t32[e] = (float)t[e];
    PR_CUDA_TRY(cudaDeviceSynchronize());
    PR_CUDA_TRY(cudaMemcpy(ctx->d_corr64, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice));
    PR_CUDA_TRY(cudaMemcpy(ctx->d_corr32, t32.data(), t32.size() * sizeof(float), cudaMemcpyHostToDevice));
    ctx->corr_nT = nT;
    ctx->corr_nP = nP;
    return PR_OK;
}

pr_status pr_set_bilger(pr_ctx *ctx, const int32_t *atoms, const double *Y_fuel, const double *Y_ox)
{
    PR_CHECK_ARG(ctx != nullptr && atoms != nullptr && Y_fuel != nullptr && Y_ox != nullptr,
                 "pr_set_bilger: null argument");
    const int N = ctx->n_species;
    // species molar masses back from the device records (1 / inv_W, kg -> g)
    std::vector<prk::SpeciesRec<double>> sp(ctx->ns_pad);
    PR_CUDA_TRY(cudaMemcpy(sp.data(), ctx->d_sp64, sp.size() * sizeof(sp[0]), cudaMemcpyDeviceToHost));
    // [N] coefficients b_k, then beta_ox and 1 / (beta_fuel - beta_ox)
    std::vector<double> packed(N + 2, 0.0);
    double bf = 0.0, bo = 0.0;
    for (int k = 0; k < N; ++k) {
        PR_CHECK_ARG(atoms[3 * k] >= 0 && atoms[3 * k + 1] >= 0 && atoms[3 * k + 2] >= 0,
                     "pr_set_bilger: negative atom count for species %d", k);
        PR_CHECK_ARG(std::isfinite(Y_fuel[k]) && std::isfinite(Y_ox[k]), "pr_set_bilger: stream not finite");
        const double Wg = 1e3 / sp[k].inv_W;
        // beta = 2 n_C + n_H / 2 - n_O, n_e = sum_k a_ek Y_k / W_k (moles of element per gram)
        packed[k] = (2.0 * atoms[3 * k] + 0.5 * atoms[3 * k + 1] - 1.0 * atoms[3 * k + 2]) / Wg;
        bf += packed[k] * Y_fuel[k];
        bo += packed[k] * Y_ox[k];
    }
    PR_CHECK_ARG(bf != bo, "pr_set_bilger: fuel and oxidiser streams have the same coupling function");
    packed[N] = bo;
    packed[N + 1] = 1.0 / (bf - bo);
    std::vector<float> p32(packed.begin(), packed.end());
    PR_CUDA_TRY(cudaDeviceSynchronize());
    PR_CUDA_TRY(cudaMemcpy(ctx->d_bilger64, packed.data(), packed.size() * sizeof(double), cudaMemcpyHostToDevice));
    PR_CUDA_TRY(cudaMemcpy(ctx->d_bilger32, p32.data(), p32.size() * sizeof(float), cudaMemcpyHostToDevice));
    ctx->has_bilger = 1;
    return PR_OK;
}

pr_status pr_bilger_z(pr_ctx *ctx, pr_precision prec, int64_t n, const void *Y, int64_t ldY, void *Z, void *stream)
{
    PR_CHECK_ARG(ctx != nullptr, "pr_bilger_z: null context");
    PR_CHECK_ARG(ctx->has_bilger, "pr_bilger_z: no element table set (pr_set_bilger)");
    PR_CHECK_ARG(prec == PR_FP64 || prec == PR_FP32 || prec == PR_MIXED, "pr_bilger_z: bad precision %d", (int)prec);
    PR_CHECK_ARG(n >= 0, "pr_bilger_z: n < 0");
    if (n == 0) return PR_OK;
    PR_CHECK_ARG(ldY >= n, "pr_bilger_z: ldY < n");
    const size_t esz = (prec == PR_FP64) ? 8 : 4;
    PR_CHECK_ARG(Y != nullptr && Z != nullptr, "pr_bilger_z: null array");
    PR_CHECK_ARG(prgb::aligned(Y, esz) && prgb::aligned(Z, esz), "pr_bilger_z: array not aligned to %zu bytes", esz);
    int64_t need = (n + kSpBlock - 1) / kSpBlock;
    const int64_t cap = (int64_t)ctx->num_sms * 16;
    const int g = (int)(need < cap ? need : cap);
    cudaStream_t st = (cudaStream_t)stream;
    if (prec == PR_FP64)
        bilger_kernel<double><<<g, kSpBlock, 0, st>>>(n, (const double *)Y, ldY, ctx->n_species, ctx->d_bilger64,
                                                      (double *)Z);
    else
        bilger_kernel<float><<<g, kSpBlock, 0, st>>>(n, (const float *)Y, ldY, ctx->n_species, ctx->d_bilger32,
                                                     (float *)Z);
    PR_CUDA_TRY(cudaGetLastError());
    return PR_OK;
}

pr_status pr_species_props(pr_ctx *ctx, pr_precision prec, int64_t n, const void *T, const void *p, const void *Y,
                           int64_t ldY, void *hk_RT, void *Dk, int64_t ldo, int32_t *cell_status, void *stream)
{
    PR_CHECK_ARG(ctx != nullptr, "pr_species_props: null context");
    PR_CHECK_ARG(prec == PR_FP64 || prec == PR_FP32 || prec == PR_MIXED, "pr_species_props: bad precision %d",
                 (int)prec);
    PR_CHECK_ARG(n >= 0, "pr_species_props: n < 0");
    if (n == 0) return PR_OK;
    PR_CHECK_ARG(ldY >= n, "pr_species_props: ldY (%lld) < n (%lld)", (long long)ldY, (long long)n);
    PR_CHECK_ARG((hk_RT == nullptr && Dk == nullptr) || ldo >= n, "pr_species_props: ldo (%lld) < n (%lld)",
                 (long long)ldo, (long long)n);
    const size_t esz = (prec == PR_FP64) ? 8 : 4;
    for (const void *q : {T, p, Y}) {
        PR_CHECK_ARG(q != nullptr, "pr_species_props: required array is NULL");
        PR_CHECK_ARG(prgb::aligned(q, esz), "pr_species_props: array not aligned to %zu bytes", esz);
    }
    for (const void *q : {hk_RT, Dk})
        PR_CHECK_ARG(prgb::aligned(q, esz), "pr_species_props: array not aligned to %zu bytes", esz);
    PR_CHECK_ARG(prgb::aligned(cell_status, 4), "pr_species_props: cell_status misaligned");
    cudaStream_t st = (cudaStream_t)stream;
    const bool nine = ctx->ns_pad == 9;
    if (prec == PR_FP64) {
        SpArgs<double> a{n, ldY, ldo, (const double *)T, (const double *)p, (const double *)Y, (double *)hk_RT,
                         (double *)Dk, cell_status, (const SpeciesRec<double> *)ctx->d_sp64, ctx->d_dtab64,
                         ctx->d_corr64, ctx->n_species, ctx->corr_nT, ctx->corr_nP};
        // the fixed-point kernel: tables within its ranges, no correction table
        if (nine && ctx->h_spfix && ctx->corr_nT == 0) {
            const int64_t need = (n + kSpBlock - 1) / kSpBlock, cap = (int64_t)ctx->occ_spfix * ctx->num_sms;
            species_fix_kernel<<<(int)(need < cap ? need : cap), kSpBlock, 0, st>>>(
                a, *static_cast<const SpFix9 *>(ctx->h_spfix));
        } else if (nine) launch_species<double, 9>(a, ctx->occ_species[0], ctx->num_sms, st);
        else launch_species<double, 32>(a, ctx->occ_species[0], ctx->num_sms, st);
    } else {
        SpArgs<float> a{n, ldY, ldo, (const float *)T, (const float *)p, (const float *)Y, (float *)hk_RT,
                        (float *)Dk, cell_status, (const SpeciesRec<float> *)ctx->d_sp32, ctx->d_dtab32,
                        ctx->d_corr32, ctx->n_species, ctx->corr_nT, ctx->corr_nP};
        if (nine) {
            const int64_t need = (n + kSpBlock - 1) / kSpBlock, cap = (int64_t)ctx->occ_species[1] * ctx->num_sms;
            species_share_kernel<<<(int)(need < cap ? need : cap), kSpBlock, 0, st>>>(
                a, *static_cast<const SpShare9 *>(ctx->h_spshare));
        }
        else launch_species<float, 32>(a, ctx->occ_species[1], ctx->num_sms, st);
    }
    PR_CUDA_TRY(cudaGetLastError());
    return PR_OK;
}

}  // extern "C"
