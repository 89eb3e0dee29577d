// The FP64 inversion kernel of contexts that take the fixed-point evaluation
// (pr_fix9.cuh).
#include "pr_fix9.cuh"

namespace prk {

// A cell of the inversion's queue through the safeguarded iteration (from its
// first evaluation when it has one), general form.
static __device__ __noinline__ void newton_finish9(const NewtonArgs<double> &a, int64_t i, double T0, bool first,
                                                   double h0, double cp0)
{
    Comp<double, 9> c;
    double Tres = M<double>::nan(), cp_last;
    int it = 0, st = kBadInput;
    if (load_comp<double, 9>(c, a.Y, a.ldY, i, a.N, a.sp))
        st = newton_solve<double, double, 9, false>(c, __ldg(a.hstar + i), __ldg(a.p + i), T0, a.sp, a.kij, a.tmid_u,
                                                    a.max_iter, a.rtol, 1e-6, Tres, it, cp_last, first, h0, cp0);
    a.Tout[i] = Tres;
    a.status[i] = st;
    if (a.iters) a.iters[i] = it;
}

// newton_fp64_queued (pr_kernels.cuh) with the first FP64 evaluation in fixed
// point; the FP32 warm start takes its mole fractions from the same limbs.
// 2.1 M cells of the flame field: 1643 -> 1155 us (345 -> 126 FP64-pipe
// instructions per cell, the pipe 74 -> 39 % busy; what holds it now is
// instruction fetch, 4.4 of 9 stall cycles per issue).
__global__ void __launch_bounds__(kBlock, 4) newton_fix_kernel(const __grid_constant__ NewtonArgs<double> a,
                                                            const __grid_constant__ Fix9 t)
{
    __shared__ Smem<float, 9, false> s32;
    __shared__ int q_n;
    __shared__ int64_t q_i[2 * kBlock];
    __shared__ double q_T[2 * kBlock], q_h[2 * kBlock], q_cp[2 * kBlock];
    __shared__ unsigned char q_first[2 * kBlock];
    if (threadIdx.x == 0) q_n = 0;
    stage<float, 9, false>(s32, a.sp32, a.pair32, a.kij32);   // ends with a barrier
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < a.n; base += stride) {
        const int64_t i = base + threadIdx.x;
        if (i < a.n) {
            const double hs = __ldg(a.hstar + i), p = __ldg(a.p + i), Tg = __ldg(a.Tg + i);
            double y[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) y[k] = (k < a.N) ? __ldg(a.Y + (int64_t)k * a.ldY + i) : 0.0;
            Fix9Comp c;
            const int ok = fix9_comp(t, y, c);
            if (ok == kFixBad || !(isfinite(hs) && isfinite(Tg) && p > 0.0 && isfinite(p))) {
                a.Tout[i] = M<double>::nan();
                a.status[i] = kBadInput;
                if (a.iters) a.iters[i] = 0;
            } else {
                double T = fmin(fmax(Tg, kTLo), kTHi);
                bool accepted = false, first = false;
                double h0 = 0.0, cp0 = 0.0;
                if (ok == kFixOk) {
                    Comp<float, 9> cf;
                    float bm = 0.f;
#pragma unroll
                    for (int k = 0; k < 9; ++k) {
                        cf.x[k] = (float)c.xh[k] * 4.6566128730773926e-10f;   // 2^-31
                        bm = fmaf(cf.x[k], s32.sp[k].b, bm);
                    }
                    cf.Wbar = (float)c.Wbar;
                    cf.bm = bm;
                    bool wok;
                    float cp32;
                    T = warm_start_fp32<9, false>(cf, T, hs, p, s32.sp, s32.kij, (float)a.tmid_u, wok, cp32);
                    if (wok && cp32 > 0.f && fix9_range(T)) {
                        Thermo<double> th;
                        fix9_thermo(t, c, T, p, th);
                        if (th.status != kNoRoot) {
                            FirstEval f;
                            f.status = th.status;
                            f.nroots = th.nroots;
                            f.h = th.h;
                            f.cp = (double)cp32;
                            f.cv_ig = (float)th.cv_ig_molar;
                            const double dT = m64::div(hs - f.h, f.cp);
                            if (one_step_ok<9>(f, T, dT, c.Wbar, s32.sp, (float)a.tmid_u)) {
                                a.Tout[i] = T + dT;
                                a.status[i] = kOk;
                                if (a.iters) a.iters[i] = 1;
                                accepted = true;
                            } else {
                                first = true;
                                h0 = f.h;
                                cp0 = f.cp;
                            }
                        }
                    }
                }
                if (!accepted) {
                    const int e = atomicAdd(&q_n, 1);
                    q_i[e] = i;
                    q_T[e] = T;
                    q_h[e] = h0;
                    q_cp[e] = cp0;
                    q_first[e] = first ? 1 : 0;
                }
            }
        }
        __syncthreads();
        while (q_n >= (int)blockDim.x) {
            const int e = q_n - (int)blockDim.x + (int)threadIdx.x;
            newton_finish9(a, q_i[e], q_T[e], q_first[e] != 0, q_h[e], q_cp[e]);
            __syncthreads();
            if (threadIdx.x == 0) q_n -= (int)blockDim.x;
            __syncthreads();
        }
    }
    if ((int)threadIdx.x < q_n) {
        const int e = threadIdx.x;
        newton_finish9(a, q_i[e], q_T[e], q_first[e] != 0, q_h[e], q_cp[e]);
    }
}

void launch_newton_fix(const NewtonArgs<double> &a, const Fix9 &t, int occ, int sms, cudaStream_t st)
{
    newton_fix_kernel<<<grid_for(a.n, occ, sms), kBlock, 0, st>>>(a, t);
}

int occupancy_newton_fix()
{
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, newton_fix_kernel, kBlock, 0);
    return occ > 0 ? occ : 1;
}

}  // namespace prk
