// The FP64 inversion kernel of contexts that take the fixed-point evaluation
// (pr_fix9.cuh).
#include "pr_fix9.cuh"

namespace prk {

// What a queued cell brings beside its start: nothing, its first evaluation,
// or the FP32 cp at a warm root outside the fixed-point range.  (Evaluated where
// it is found, such a root holds back its warp's other cells: 300000 cells, one
// in six above 4096 K, 471 us, queued 372.)
enum QueuedAs : unsigned char { kStartOnly = 0, kEvaluated = 1, kWarmRoot = 2 };

// A cell of the inversion's queue, general form: one evaluation at a warm
// root and the one-step acceptance, else the safeguarded iteration (from the
// first evaluation when there is one).
static __device__ __noinline__ void newton_finish9(const NewtonArgs<double> &a, const SpeciesRec<float> *sp32, int64_t i,
                                                   double T0, int as, double h0, double cp0)
{
    Comp<double, 9> c;
    double Tres = M<double>::nan(), cp_last;
    int it = 0, st = kBadInput;
    if (load_comp<double, 9>(c, a.Y, a.ldY, i, a.N, a.sp)) {
        const double hs = __ldg(a.hstar + i), p = __ldg(a.p + i);
        bool accepted = false;
        if (as == kWarmRoot) {
            FirstEval f = eval_h_first<double, double, 9, false>(c, T0, p, a.sp, a.kij, a.tmid_u);
            if (f.status == kNoRoot) {
                as = kStartOnly;
            } else {
                f.cp = cp0;
                h0 = f.h;
                const double dT = m64::div(hs - f.h, f.cp);
                if (one_step_ok<9>(f, T0, dT, c.Wbar, sp32, (float)a.tmid_u)) {
                    accepted = true;
                    Tres = T0 + dT;
                    st = kOk;
                    it = 1;
                }
            }
        }
        if (!accepted)
            st = newton_solve<double, double, 9, false>(c, hs, p, T0, a.sp, a.kij, a.tmid_u, a.max_iter, a.rtol, 1e-6,
                                                        Tres, it, cp_last, as != kStartOnly, h0, cp0);
    }
    a.Tout[i] = Tres;
    a.status[i] = st;
    if (a.iters) a.iters[i] = it;
}

// The inversion in two launches: in one kernel the FP32 iterations and the
// FP64 evaluation missed the instruction cache (half of the stall cycles) and
// ran at the FP64 part's 128 registers.  First the FP32 warm start of every cell, T
// into Tout and the FP32 cp at it, as bits, into the status array (0 where
// the warm start failed: T is then the clamped guess; -1: a guess refused) ...
__global__ void __launch_bounds__(kBlock) newton_warm_kernel(const __grid_constant__ NewtonArgs<double> a,
                                                             const __grid_constant__ ParamTab<float, 9, false> t,
                                                             const __grid_constant__ WarmTab w)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
        const float hs = (float)__ldg(a.hstar + i), p = (float)__ldg(a.p + i);
        const double Tg = a.Tg[i];   // Tg may be Tout
        const double T0 = fmin(fmax(Tg, kTLo), kTHi);
        double y[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) y[k] = (k < a.N) ? __ldg(a.Y + (int64_t)k * a.ldY + i) : 0.0;
        Comp<float, 9> c;
        warm_comp(w, y, c);
        // warm_start_fp32's iteration with its evaluations at one place, in
        // line, the tables as constant operands (states refused by the second
        // launch pass through here too: the loop is bounded)
        float T = (float)T0, cp_end = 0.f;
        bool ok = false;
#pragma unroll 1
        for (int k = 0; k < 9; ++k) {
            Thermo<float> th;
            thermo<float, float, 9, false>(c, T, p, t.sp, t.kij, th, (float)a.tmid_u);
            if (th.status == kNoRoot || !(th.cp > 0.f)) break;
            if (ok) {   // the step before was the last one: cp at the root
                cp_end = th.cp;
                break;
            }
            const float Tn = T - (th.h - hs) / th.cp;
            if (!(Tn > (float)kTLo && Tn < (float)kTHi) || k == 8) break;
            ok = fabsf(Tn - T) <= 1e-5f * Tn;
            T = Tn;
        }
        a.Tout[i] = cp_end > 0.f ? (double)T : T0;
        a.status[i] = __float_as_int(isfinite(Tg) ? cp_end : -1.f);
    }
}

// ... then one FP64 evaluation per cell, in fixed point, and the one-step
// acceptance; the other cells through a queue of the block, as
// newton_fp64_queued (pr_kernels.cuh).
__device__ __forceinline__ void newton_fix_cell(const NewtonArgs<double> &a, const Fix9 &t, int64_t i, double T,
                                                float cp32, const SpeciesRec<float> *sp32, int *q_n,
                                                int64_t *q_i, double *q_T, double *q_h, double *q_cp,
                                                unsigned char *q_as, bool guess_ok)
{
    const double hs = __ldg(a.hstar + i), p = __ldg(a.p + i);
    double y[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) y[k] = (k < a.N) ? __ldg(a.Y + (int64_t)k * a.ldY + i) : 0.0;
    Fix9Comp c;
    const int ok = fix9_comp(t, y, c);
    if (ok == kFixBad || !(guess_ok && isfinite(hs) && p > 0.0 && isfinite(p))) {
        a.Tout[i] = M<double>::nan();
        a.status[i] = kBadInput;
        if (a.iters) a.iters[i] = 0;
        return;
    }
    int as = cp32 > 0.f ? kWarmRoot : kStartOnly;
    double h0 = 0.0, cp0 = (double)cp32;
    if (ok == kFixOk && cp32 > 0.f && fix9_range(T)) {
        Thermo<double> th;
        fix9_thermo(t, c, T, p, th);
        as = kStartOnly;
        // the acceptance's table loads stay below the evaluation, whose registers
        // they would take (2.1 M cells 698 us without this line, 642 with it)
        asm volatile("" ::: "memory");
        if (th.status != kNoRoot) {
            FirstEval f;
            f.status = th.status;
            f.nroots = th.nroots;
            f.h = th.h;
            f.cp = cp0;
            f.cv_ig = (float)th.cv_ig_molar;
            const double dT = m64::div(hs - f.h, f.cp);
            if (one_step_ok<9>(f, T, dT, c.Wbar, sp32, (float)a.tmid_u)) {
                a.Tout[i] = T + dT;
                a.status[i] = kOk;
                if (a.iters) a.iters[i] = 1;
                return;
            }
            as = kEvaluated;
            h0 = f.h;
        }
    }
    const int e = atomicAdd(q_n, 1);
    q_i[e] = i;
    q_T[e] = T;
    q_h[e] = h0;
    q_cp[e] = cp0;
    q_as[e] = (unsigned char)as;
}

// SPLIT: T and cp from newton_warm_kernel; else the warm start runs here.
template <bool SPLIT>
__global__ void __launch_bounds__(kBlock, 4) newton_fix_kernel(const __grid_constant__ NewtonArgs<double> a,
                                                               const __grid_constant__ Fix9 t)
{
    __shared__ Smem<float, 9, false> s32;
    __shared__ int q_n;
    __shared__ int64_t q_i[2 * kBlock];
    __shared__ double q_T[2 * kBlock], q_h[2 * kBlock], q_cp[2 * kBlock];
    __shared__ unsigned char q_as[2 * kBlock];
    if (threadIdx.x == 0) q_n = 0;
    stage<float, 9, false>(s32, a.sp32, a.pair32, a.kij32);   // ends with a barrier
    auto finish = [&](int e) { newton_finish9(a, s32.sp, q_i[e], q_T[e], q_as[e], q_h[e], q_cp[e]); };
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < a.n; base += stride) {
        const int64_t i = base + threadIdx.x;
        if (i < a.n) {
            if constexpr (SPLIT) {
                const float cp32 = __int_as_float(a.status[i]);
                newton_fix_cell(a, t, i, a.Tout[i], cp32, s32.sp, &q_n, q_i, q_T, q_h, q_cp, q_as, cp32 >= 0.f);
            } else {
                const double Tg = __ldg(a.Tg + i);
                double y[9];
#pragma unroll
                for (int k = 0; k < 9; ++k) y[k] = (k < a.N) ? __ldg(a.Y + (int64_t)k * a.ldY + i) : 0.0;
                Comp<float, 9> cf;
                warm_comp(t.warm, y, cf);
                bool wok;
                float cp32;
                const double T = warm_start_fp32<9, false>(cf, fmin(fmax(Tg, kTLo), kTHi), __ldg(a.hstar + i),
                                                           __ldg(a.p + i), s32.sp, s32.kij, (float)a.tmid_u, wok, cp32);
                newton_fix_cell(a, t, i, T, wok ? cp32 : 0.f, s32.sp, &q_n, q_i, q_T, q_h, q_cp, q_as, isfinite(Tg));
            }
        }
        queue_round(&q_n, (int)threadIdx.x, (int)blockDim.x, finish);
    }
    queue_rest(&q_n, (int)threadIdx.x, finish);
}

// [a, a + na) and [b, b + nb) share a byte
static bool overlap(const void *a, size_t na, const void *b, size_t nb)
{
    const char *x = static_cast<const char *>(a), *y = static_cast<const char *>(b);
    return x < y + nb && y < x + na;
}

void launch_newton_fix(const NewtonArgs<double> &a, const Fix9 &t, const void *htab32, const int occ[3], int sms,
                       cudaStream_t st)
{
    // the first launch writes Tout and status: only the guess may be among
    // them (element by element), not what the second launch reads
    const size_t nb = (size_t)a.n * 8, yb = ((size_t)a.ldY * (size_t)(a.N - 1) + (size_t)a.n) * 8;
    const bool own = !overlap(a.Tout, nb, a.hstar, nb) && !overlap(a.Tout, nb, a.p, nb) && !overlap(a.Tout, nb, a.Y, yb) &&
                     (a.Tout == a.Tg || !overlap(a.Tout, nb, a.Tg, nb)) && !overlap(a.status, nb / 2, a.Tout, nb) &&
                     !overlap(a.status, nb / 2, a.hstar, nb) && !overlap(a.status, nb / 2, a.p, nb) &&
                     !overlap(a.status, nb / 2, a.Y, yb) && !overlap(a.status, nb / 2, a.Tg, nb);
    // two launches for more cells than one wave of the single kernel holds:
    // up to there the second launch costs more than the smaller kernels gain
    // (65536 cells, in one wave: 63 us against 65; 131072: 107 against 82;
    // 2.1 M cells: 1176 against 641)
    if (a.n > (int64_t)occ[2] * sms * kBlock && own) {
        newton_warm_kernel<<<grid_for(a.n, occ[0], sms), kBlock, 0, st>>>(a, make_tab<float, 9, false>(htab32), t.warm);
        newton_fix_kernel<true><<<grid_for(a.n, occ[1], sms), kBlock, 0, st>>>(a, t);
    } else {
        const int b = block_for(a.n, sms);
        newton_fix_kernel<false><<<grid_for(a.n, occ[2], sms, b), b, 0, st>>>(a, t);
    }
}

void occupancy_newton_fix(int occ[3])
{
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[0], newton_warm_kernel, kBlock, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[1], newton_fix_kernel<true>, kBlock, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[2], newton_fix_kernel<false>, kBlock, 0);
    for (int k = 0; k < 3; ++k) occ[k] = occ[k] > 0 ? occ[k] : 1;
}

}  // namespace prk
