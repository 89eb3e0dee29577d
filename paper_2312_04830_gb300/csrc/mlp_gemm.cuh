// Tensor-core GEMM for the surrogate MLP: D[M x N] = A[M x K] * B[N x K]^T
// with BF16 operands (both K-major, loaded by TMA with 128-byte swizzling),
// FP32 accumulators in tensor memory (tcgen05.mma: M = 128 a CTA, or 256 on a
// pair of CTAs) and fused epilogues for every GEMM of the MLP's forward and
// backward pass.
//
// Persistent kernel, one CTA per SM, 18 warps (the plain GEMM 10): warp 0
// issues TMA loads into an S-stage shared-memory ring, one thread of warp 1
// issues the MMAs (K = 16 each, 4 per 64-wide k-block), the other warps drain
// the accumulator and run the epilogue (warp w owns TMEM lane quarter w % 4,
// i.e. 32 rows, and a quarter, in the plain GEMM a half, of the tile's columns).  The accumulator is double-buffered in TMEM (2 x BN
// columns), so the epilogue of one tile overlaps the main loop of the next.
// Tiles are visited with the N index fastest, so the N-tiles of one M-tile run
// together and share the A tile through L2.  A pair takes two adjacent M-tiles
// and each of its CTAs loads half of the B tile: 32 KB a k-block and CTA where
// a single CTA loads 48.
//
// Per 65536 x 512 x 512 GEMM of a training step, us, in the step (8 epilogue
// warps and single CTAs | 16 warps and pairs): hidden layer 48 | 46, input
// gradient 54 | 50, weight gradient 39 | 33; with K = 64, on single CTAs with
// 16 warps too, hidden 34 | 27 and input gradient 48 | 32.  What is left above the MMAs' 15 us: 8 to 10 us to
// launch, fill and drain, and the epilogue's traffic, which slows the main
// loop (a hidden layer's takes 27 us without an epilogue, 36 without its
// stores and 42 without the GeLU).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "umma.cuh"

namespace mlp {

constexpr int BM = 128;
constexpr int BK = 64;

enum Epi : int {
    kEpiHidden = 0,    // h = GeLU(acc + b) -> out; (train) GeLU'(acc + b) -> gd
    kEpiOutPhys = 1,   // y = acc + b (n < nout) -> de-standardise -> physical values out6[nout][ld6]
    kEpiOutLoss = 2,   // y = acc + b; d = y - target (0 where the target is not finite); loss += d^2 (or |d|);
                       // dz = scale d -> out, colsum
    kEpiDx = 3,        // dz = acc * gd -> out, colsum
    kEpiDw = 4,        // partial[split][m][n] = acc (FP32)
    kEpiDwMN = 5,      // as kEpiDw, with A and B read MN-major: A from [K][M], B from [K][N]
                       // (tmA / tmB with 64 x 64 boxes), e.g. dW = dz^T h from the batch-major dz
                       // and h; BN >= 64
};

struct GemmArgs {
    int M, N, K;              // logical sizes; A is [M][K], B is [N][K]
    int kb_per_split;         // 64-wide k-blocks per K split
    int m_tiles, n_tiles, splits;   // tile grid (splits along K)
    const float *bias;        // [N]
    __nv_bfloat16 *out;       // kEpiOutLoss: dz [M][ldo] batch-major
    int64_t ldo;
    float *partial;           // kEpiDw: [split][Mpad][N]
    int Mpad;
    float *colsum;            // [m_tiles][N] per-M-tile column sums of dz (bias gradients)
    float *out6;              // kEpiOutPhys: [nout][ld6]
    int64_t ld6;
    const float *out_mean, *out_std;   // [nout] de-standardisation
    const float *add_h;       // kEpiOutPhys: per-row term added to output 2 (h) after de-standardisation
    int log_mask;             // kEpiOutPhys: bit j set = output j was learned as its logarithm
    const float *target;      // kEpiOutLoss: standardised targets [nout][ldt]
    int64_t ldt;
    float loss_scale;         // d loss / d y = loss_scale * (y - target), or loss_scale * sign(y - target) (l1)
    float *loss_part;         // [m_tiles] per-M-tile sum of squared (l1: absolute) errors
    int l1;                   // kEpiOutLoss: 1 = L1 loss, 0 = squared error
    int nout;                 // kEpiOutPhys / kEpiOutLoss: outputs in use (<= 16)
    int *err;                 // set to 1 when a bounded wait runs out
    // kEpiHidden / kEpiDx: the output (h or dz) and GeLU'(z) (written by
    // kEpiHidden when `train` is set, read by kEpiDx), both [M][N] batch-major,
    // go through shared memory and TMA boxes of 32 x 32 (64-byte swizzle)
    int train;
    // L2 (an activation matrix of 65536 x 512 is half of it): A and B leave
    // first after their loads here, if this is their last use for long, as
    // GeLU'(z) always does, and M-tiles go in descending order (flip) after a
    // GEMM whose output, A here, was written in ascending order.  A hidden
    // layer then finds its input in L2 (DRAM reads 67 -> 9 MB), a weight
    // gradient its dz (134 -> 77 MB).
    int last_a, last_b, flip;
    CUtensorMap tm_out, tm_gd;
};

// Epilogue warps: 16, but 8 for the plain GEMM, whose FP32 rows the store units
// hold (65536 x 512 x 64: 47.5 us with 16, 44.4 with 8; x 512 60.9 and 57.4).
constexpr int epi_warps(int EPI) { return EPI == kEpiDw ? 8 : 16; }

// Rows of B per TMA box of a K-major GEMM: the half that one CTA of a pair
// loads (a single CTA loads two boxes, one above the other).
constexpr int b_box_rows(int BN) { return BN >= 128 ? BN / 2 : BN; }

template <int BN, int EPI, bool PAIR>
struct Cfg {
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int B_BYTES = (PAIR ? BN / 2 : BN) * BK * 2;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int WARPS = epi_warps(EPI);
    static constexpr int THREADS = 64 + 32 * WARPS;
    static constexpr bool SPLIT_N = BN >= 4 * WARPS;                    // each quarter's warps share the columns
    static constexpr int COLS = SPLIT_N ? BN / (WARPS / 4) : BN;   // columns per epilogue warp
    // output staging, two 2 KB boxes per epilogue warp.  (Without any, the
    // weight gradients have six stages for four: 36 -> 33 us.)
    static constexpr int STG_BYTES = (EPI == kEpiHidden || EPI == kEpiDx) ? WARPS * 4096 : 0;
    static constexpr int S_FIT = (232448 - 1024 - STG_BYTES - 13312) / STAGE;
    static constexpr int S = S_FIT < 8 ? S_FIT : 8;
    static constexpr uint32_t TMEM_COLS = (2 * BN) < 32 ? 32 : 2 * BN;   // two accumulator buffers
    static constexpr int BAR_BYTES = 8 * (2 * S + 5 + 2 * WARPS) + 24;
    static constexpr int RED_FLOATS = 4 * BN + 16;          // one tile's column sums and loss sums; two tiles' worth
    static constexpr int RED_BYTES = 2 * RED_FLOATS * 4;
    static constexpr int BIAS_BYTES = 1024 * 4;   // bias of up to 1024 output columns
    static constexpr int SMEM = 1024 + S * STAGE + STG_BYTES + BAR_BYTES + RED_BYTES + BIAS_BYTES;
    static_assert(SMEM <= 232448 && BAR_BYTES % 16 == 0, "shared memory");
};

// GeLU in its tanh form (Hendrycks & Gimpel 2016),
//   GeLU(z) ~ z/2 (1 + tanh(k (z + c z^3))),  k = sqrt(2/pi), c = 0.044715,
// with the hardware tanh.approx.f32 (one MUFU operation), and its exact
// derivative
//   GeLU'(z) = (1 + t)/2 + z/2 (1 - t^2) k (1 + 3 c z^2),  t = tanh(k (z + c z^3)).
// The tanh form differs from z Phi(z) by at most 5e-4 and tanh.approx has a
// relative error below 2^-10.9; both are under the BF16 rounding of the
// activations (3.9e-3).  Training and inference use this same function.
__device__ __forceinline__ float tanh_approx(float x)
{
    float r;
    asm("tanh.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

constexpr float kGeluK = 0.7978845608028654f;            // sqrt(2/pi)
constexpr float kGeluKC = 0.7978845608028654f * 0.044715f;

__device__ __forceinline__ float gelu_f(float z)
{
    const float z2 = z * z;
    const float t = tanh_approx(z * fmaf(kGeluKC, z2, kGeluK));
    const float hz = 0.5f * z;
    return fmaf(hz, t, hz);
}

// gelu_f of z = a + b on two lanes at once with the packed FP32 instructions
// of sm_100 (FADD2 / FMUL2 / FFMA2): the same operations in the same order as
// gelu_f(a + b), so the same bits, in about half the FP32 instructions.
__device__ __forceinline__ float2 gelu2(float2 a, float2 b)
{
    const float2 z = __fadd2_rn(a, b);
    const float2 z2 = __fmul2_rn(z, z);
    const float2 p = __ffma2_rn(make_float2(kGeluKC, kGeluKC), z2, make_float2(kGeluK, kGeluK));
    const float2 u = __fmul2_rn(z, p);
    const float2 t = make_float2(tanh_approx(u.x), tanh_approx(u.y));
    const float2 hz = __fmul2_rn(make_float2(0.5f, 0.5f), z);
    return __ffma2_rn(hz, t, hz);
}

// GeLU(z) and GeLU'(z) of z = a + b on two lanes at once (packed FP32).
__device__ __forceinline__ void gelu_and_grad2(float2 a, float2 b, float2 &g, float2 &dg)
{
    const float2 z = __fadd2_rn(a, b);
    const float2 z2 = __fmul2_rn(z, z);
    const float2 u = __fmul2_rn(z, __ffma2_rn(make_float2(kGeluKC, kGeluKC), z2, make_float2(kGeluK, kGeluK)));
    const float2 t = make_float2(tanh_approx(u.x), tanh_approx(u.y));
    const float2 hz = __fmul2_rn(make_float2(0.5f, 0.5f), z);
    g = __ffma2_rn(hz, t, hz);
    const float2 dk = __ffma2_rn(make_float2(3.0f * kGeluKC, 3.0f * kGeluKC), z2, make_float2(kGeluK, kGeluK));
    const float2 omt = __ffma2_rn(make_float2(-t.x, -t.y), t, make_float2(1.0f, 1.0f));
    dg = __ffma2_rn(__fmul2_rn(hz, omt), dk, __ffma2_rn(make_float2(0.5f, 0.5f), t, make_float2(0.5f, 0.5f)));
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ void store_row16_bf16(__nv_bfloat16 *dst, const float (&v)[16])
{
    uint4 lo = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    uint4 hi = make_uint4(pack_bf16(v[8], v[9]), pack_bf16(v[10], v[11]), pack_bf16(v[12], v[13]),
                          pack_bf16(v[14], v[15]));
    reinterpret_cast<uint4 *>(dst)[0] = lo;
    reinterpret_cast<uint4 *>(dst)[1] = hi;
}

// 16 BF16 of row `row` (0..31), columns 16*c .. 16*c+15, into a staging box of
// 32 rows x BC columns laid out as TMA's 128-byte (BC = 64: the 16-byte piece
// j of row r at piece j ^ (r % 8)) or 64-byte swizzle (BC = 32: j ^ (r/2 % 4)).
template <int BC = 64>
__device__ __forceinline__ void stage_row16_bf16(uint8_t *box, int row, int c, const float (&v)[16])
{
    static_assert(BC == 64 || BC == 32, "boxes of one swizzle row");
    const uint4 lo = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                                pack_bf16(v[6], v[7]));
    const uint4 hi = make_uint4(pack_bf16(v[8], v[9]), pack_bf16(v[10], v[11]), pack_bf16(v[12], v[13]),
                                pack_bf16(v[14], v[15]));
    uint8_t *r = box + row * (BC * 2);
    const int j0 = 2 * c, x = (BC == 64) ? row & 7 : (row >> 1) & 3;
    *reinterpret_cast<uint4 *>(r + ((j0 ^ x) << 4)) = lo;
    *reinterpret_cast<uint4 *>(r + (((j0 + 1) ^ x) << 4)) = hi;
}

// 16 BF16 of a staging box of 32 x 32 (as stage_row16_bf16<32> places them)
__device__ __forceinline__ void unstage_row16_bf16(const uint8_t *box, int row, int c, float (&v)[16])
{
    const uint8_t *r = box + row * 64;
    const int j0 = 2 * c, x = (row >> 1) & 3;
    const uint4 lo = *reinterpret_cast<const uint4 *>(r + ((j0 ^ x) << 4));
    const uint4 hi = *reinterpret_cast<const uint4 *>(r + (((j0 + 1) ^ x) << 4));
    const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[k]));
        v[2 * k] = f.x;
        v[2 * k + 1] = f.y;
    }
}

// Sum 16 per-lane values over the 32 lanes of a warp; afterwards even lane L
// holds the sum of column (L >> 1).  15 shuffles instead of 80.
__device__ __forceinline__ float warp_colsum16(float (&v)[16], int lane)
{
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const bool up = lane & 16;
        const float send = up ? v[k] : v[k + 8];
        const float keep = up ? v[k + 8] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool up = lane & 8;
        const float send = up ? v[k] : v[k + 4];
        const float keep = up ? v[k + 4] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const bool up = lane & 4;
        const float send = up ? v[k] : v[k + 2];
        const float keep = up ? v[k + 2] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    {
        const bool up = lane & 2;
        const float send = up ? v[0] : v[1];
        const float keep = up ? v[1] : v[0];
        v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

template <int THREADS>
__device__ __forceinline__ void named_barrier_epi()
{
    asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// Tile `t` of the grid-stride walk: K split, M-tile index (of this CTA: a pair
// takes two adjacent M-tiles) and N offset.
template <int BN, bool PAIR>
__device__ __forceinline__ void tile_of(const GemmArgs &a, int t, int rank, int &split, int &mt, int &n0)
{
    const int mrows = PAIR ? (a.m_tiles + 1) / 2 : a.m_tiles;
    const int per_split = mrows * a.n_tiles;
    split = t / per_split;
    const int r = t % per_split;
    mt = r / a.n_tiles;
    n0 = (r % a.n_tiles) * BN;
    if (a.flip) mt = mrows - 1 - mt;
    if (PAIR) mt = 2 * mt + rank;
}

// kEpiDx: GeLU'(z) comes in as the output goes out, in boxes of 32 rows x 32
// columns in shared memory, two per warp taking turns; dz replaces GeLU'(z) in
// its box.  (Loaded per lane from global memory, a row and so a cache line
// each, the loads held the kernel: 48 us at K = 64, now 35.)
struct GradBoxes {
    uint64_t *full;      // [2]
    uint32_t nload = 0;  // (lane 0) boxes asked for
    uint32_t nuse = 0;   // boxes waited for
};

// Epilogue of one accumulator tile for one epilogue warp: drain this warp's
// 32 rows x COLS columns from TMEM, apply the epilogue, store.  Returns this
// lane's sum of squared errors (kEpiOutLoss).  `refill` (kEpiDx, lane 0) asks
// for the next GeLU'(z) box, once the stores from its place have left.
template <int BN, int EPI, class Refill>
__device__ __forceinline__ float epilogue_tile(const GemmArgs &a, uint32_t taddr, int m, bool mval, int n0, int hcol,
                                               int q, int lane, int split, float *red, const float *sbias,
                                               bool active, bool store, bool &fail, uint8_t *stg, int m0,
                                               GradBoxes &gb, Refill refill)
{
    constexpr int COLS = Cfg<BN, EPI, false>::COLS;
    constexpr bool kBoxes = EPI == kEpiHidden || EPI == kEpiDx;
    static_assert(!kBoxes || COLS % 32 == 0, "hidden layers: N tiles of 128 or 256");
    float lsum = 0.f;
    if (active && !fail) {
#pragma unroll 1
        for (int c = 0; c < COLS / 16; ++c) {
            const int nb = n0 + hcol + c * 16;
            uint8_t *box = stg;
            if (EPI == kEpiDx) box = stg + (gb.nuse & 1u) * 2048;
            if (EPI == kEpiHidden && (c & 1) == 0) {
                if (lane == 0) umma::bulk_wait_read0();
                __syncwarp();
            }
            if (EPI == kEpiDx && (c & 1) == 0) {
                if (!umma::mbar_wait(&gb.full[gb.nuse & 1u], (gb.nuse >> 1) & 1u)) fail = true;
                fail = __any_sync(0xffffffffu, fail);
            }
            uint32_t rr[16];
            umma::tmem_ld16(taddr + c * 16, rr);
            float bias[16];
            if (EPI == kEpiHidden || EPI == kEpiOutPhys || EPI == kEpiOutLoss) {
                const float4 *sb = reinterpret_cast<const float4 *>(sbias + nb);   // broadcast reads
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    const float4 b4 = sb[jj];
                    bias[4 * jj] = b4.x; bias[4 * jj + 1] = b4.y; bias[4 * jj + 2] = b4.z; bias[4 * jj + 3] = b4.w;
                }
            }
            float g[16];
            if (EPI == kEpiDx) unstage_row16_bf16(box, lane, c & 1, g);
            umma::tmem_ld_wait(rr);
            float v[16];
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) v[jj] = __uint_as_float(rr[jj]);
            if (EPI == kEpiHidden) {
                if (a.train) {
                    float gg[16];
#pragma unroll
                    for (int jj = 0; jj < 16; jj += 2) {
                        float2 g2, d2;
                        gelu_and_grad2(make_float2(v[jj], v[jj + 1]), make_float2(bias[jj], bias[jj + 1]), g2, d2);
                        v[jj] = g2.x; v[jj + 1] = g2.y;
                        gg[jj] = d2.x; gg[jj + 1] = d2.y;
                    }
                    stage_row16_bf16<32>(box + 2048, lane, c & 1, gg);
                } else {
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj) v[jj] = gelu_f(v[jj] + bias[jj]);
                }
                stage_row16_bf16<32>(box, lane, c & 1, v);
            } else if (EPI == kEpiOutPhys) {
                if (mval && nb == 0) {
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj) {
                        if (jj >= a.nout) break;
                        const float sv = v[jj] + bias[jj];
                        float qv = sv * __ldg(a.out_std + jj) + __ldg(a.out_mean + jj);
                        if (jj == 2 && a.add_h) qv += __ldg(a.add_h + m);
                        a.out6[(int64_t)jj * a.ld6 + m] = ((a.log_mask >> jj) & 1) ? __expf(qv) : qv;
                    }
                }
            } else if (EPI == kEpiOutLoss) {
#pragma unroll
                for (int jj = 0; jj < 16; ++jj) {
                    float d = 0.f;
                    if (mval && nb == 0 && jj < a.nout) {
                        const float tv = __ldg(a.target + (int64_t)jj * a.ldt + m);
                        d = isfinite(tv) ? v[jj] + bias[jj] - tv : 0.f;   // non-finite targets are masked
                    }
                    if (a.l1) {
                        lsum += fabsf(d);
                        v[jj] = a.loss_scale * (float)((d > 0.f) - (d < 0.f));
                    } else {
                        lsum += d * d;
                        v[jj] = a.loss_scale * d;
                    }
                }
                if (mval) store_row16_bf16(a.out + (int64_t)m * a.ldo + nb, v);
            } else if (EPI == kEpiDx) {
#pragma unroll
                for (int jj = 0; jj < 16; ++jj) v[jj] = mval ? v[jj] * g[jj] : 0.f;
                stage_row16_bf16<32>(box, lane, c & 1, v);
                if (c == 2 && lane == 0) refill();   // (the box of the first half: its store has had a chunk's time)
            } else {  // kEpiDw, kEpiDwMN
                if (store && m < a.Mpad) {
                    float4 *dst = reinterpret_cast<float4 *>(a.partial + ((int64_t)split * a.Mpad + m) * a.N + nb);
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj)
                        dst[jj] = make_float4(v[4 * jj], v[4 * jj + 1], v[4 * jj + 2], v[4 * jj + 3]);
                }
            }
            if (kBoxes && (c & 1) == 1) {
                umma::fence_async_smem();   // staging writes visible to the TMA engine
                __syncwarp();
                if (lane == 0 && store) {
                    umma::tma_store_2d(&a.tm_out, box, nb - 16, m0 + q * 32);
                    if (EPI == kEpiHidden && a.train) 
                        umma::tma_store_2d_hint(&a.tm_gd, box + 2048, nb - 16, m0 + q * 32, umma::l2_evict_first());
                    umma::bulk_commit();
                }
                if (EPI == kEpiDx) ++gb.nuse;
            }
            if (EPI == kEpiOutLoss || EPI == kEpiDx) {
                const float sv = warp_colsum16(v, lane);
                if ((lane & 1) == 0) red[q * BN + hcol + c * 16 + (lane >> 1)] = sv;
            }
        }
    }
    return lsum;
}

template <int BN, int EPI, bool PAIR>
__global__ void __launch_bounds__(64 + 32 * epi_warps(EPI), 1) gemm_kernel(const __grid_constant__ CUtensorMap tmA,
                                                           const __grid_constant__ CUtensorMap tmB,
                                                           const __grid_constant__ GemmArgs a)
{
    using C = Cfg<BN, EPI, PAIR>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *stg_base = smem + C::S * C::STAGE;   // 1024-aligned: stages are whole KB
    uint64_t *full = reinterpret_cast<uint64_t *>(stg_base + C::STG_BYTES);
    uint64_t *empty = full + C::S;
    uint64_t *acc_full = empty + C::S;     // [2]
    uint64_t *acc_empty = acc_full + 2;    // [2]
    uint64_t *drain = acc_empty + 2;       // (PAIR) every MMA issued has completed
    uint64_t *gfull = drain + 1;           // [WARPS][2] GeLU'(z) boxes landed
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(gfull + 2 * C::WARPS);
    float *red = reinterpret_cast<float *>(stg_base + C::STG_BYTES + C::BAR_BYTES);   // 2 x ([4][BN] + 16)
    float *sbias = red + 2 * C::RED_FLOATS;                                          // [N] (N <= 1024)

    static_assert(EPI != kEpiDwMN || BN >= 64, "MN-major operands come in 64-wide boxes");
    static_assert(!PAIR || BN >= 128, "a pair's halves of B are whole boxes");
    constexpr bool kMN = EPI == kEpiDwMN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kb_total = (a.K + BK - 1) / BK;
    const int per_split = (PAIR ? (a.m_tiles + 1) / 2 : a.m_tiles) * a.n_tiles;
    const int total = per_split * a.splits;
    const int rank = PAIR ? (int)umma::cluster_ctarank() : 0;
    const bool leader = rank == 0;
    const int t_first = PAIR ? blockIdx.x >> 1 : blockIdx.x, t_step = PAIR ? gridDim.x >> 1 : gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::S; ++s) {
            umma::mbar_init(&full[s], 1);
            umma::mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            umma::mbar_init(&acc_full[b], 1);
            umma::mbar_init(&acc_empty[b], (PAIR ? 2 : 1) * C::WARPS);
        }
        umma::mbar_init(drain, 1);
        for (int b = 0; b < 2 * C::WARPS; ++b) umma::mbar_init(&gfull[b], 1);
        umma::fence_mbar_init();
        umma::tma_prefetch_desc(&tmA);
        umma::tma_prefetch_desc(&tmB);
    }
    if (warp == 1) {
        if constexpr (PAIR) {
            umma::tmem_alloc_pair(tmem_slot, C::TMEM_COLS);
            umma::tmem_relinquish_pair();
        } else {
            umma::tmem_alloc(tmem_slot, C::TMEM_COLS);
            umma::tmem_relinquish();
        }
    }
    umma::tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) umma::cluster_sync();   // both CTAs' barriers initialised before any copy or MMA signals them
    umma::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool fail = false;
    umma::pdl_wait();      // (no global memory is touched above)
    umma::pdl_release();

    if (warp == 0) {
        // ------------------------------------------- TMA producer (each CTA)
        if (lane == 0) {
            uint32_t it = 0;
            const uint64_t pol_a = a.last_a ? umma::l2_evict_first() : umma::l2_evict_normal();
            const uint64_t pol_b = a.last_b ? umma::l2_evict_first() : umma::l2_evict_normal();
            for (int t = t_first; t < total && !fail; t += t_step) {
                int split, mt, n0;
                tile_of<BN, PAIR>(a, t, rank, split, mt, n0);
                const int m0 = mt * BM;
                const int nl = n0 + (PAIR ? rank * (BN / 2) : 0);   // this CTA's rows of B
                const int kb0 = split * a.kb_per_split;
                const int nkb = min(a.kb_per_split, kb_total - kb0);
                for (int kb = 0; kb < nkb; ++kb, ++it) {
                    const int s = it % C::S;
                    const uint32_t ph = (it / C::S) & 1u;
                    if (it >= (uint32_t)C::S && !umma::mbar_wait(&empty[s], ph ^ 1u)) { fail = true; break; }
                    uint8_t *st = smem + s * C::STAGE;
                    if (leader) umma::mbar_arrive_expect_tx(&full[s], (PAIR ? 2 : 1) * C::STAGE);
                    // (a pair's copies complete on the leader's barrier)
                    const uint32_t bar =
                        PAIR ? umma::mapa_shared(umma::smem_u32(&full[s]), 0u) : umma::smem_u32(&full[s]);
                    auto load = [&](uint8_t *dst, const CUtensorMap *tm, int c0, int c1) {
                        if constexpr (EPI == kEpiDw) {
                            // no policy beside the stores of FP32 rows: with evict_normal on
                            // the loads 65536 x 512 x 512 takes 66 us, without 57
                            if constexpr (PAIR) umma::tma_load_2d_pair(dst, tm, bar, c0, c1);
                            else umma::tma_load_2d(dst, tm, &full[s], c0, c1);
                            return;
                        }
                        const uint64_t pol = tm == &tmA ? pol_a : pol_b;
                        if constexpr (PAIR) umma::tma_load_2d_pair_hint(dst, tm, bar, c0, c1, pol);
                        else umma::tma_load_2d_hint(dst, tm, &full[s], c0, c1, pol);
                    };
                    if constexpr (kMN) {
                        // 64 k-rows of 64 M (N) columns per box; blocks of 64 columns 8 KB apart
                        const int kr = (kb0 + kb) * BK;
#pragma unroll
                        for (int i = 0; i < C::A_BYTES / 8192; ++i) load(st + i * 8192, &tmA, m0 + 64 * i, kr);
#pragma unroll
                        for (int j = 0; j < C::B_BYTES / 8192; ++j)
                            load(st + C::A_BYTES + j * 8192, &tmB, nl + 64 * j, kr);
                    } else {
                        constexpr int BR = b_box_rows(BN);
                        load(st, &tmA, (kb0 + kb) * BK, m0);
#pragma unroll
                        for (int j = 0; j < C::B_BYTES / (BR * BK * 2); ++j)
                            load(st + C::A_BYTES + j * (BR * BK * 2), &tmB, (kb0 + kb) * BK, nl + BR * j);
                    }
                }
            }
            const uint32_t it_end = it;
            if constexpr (PAIR) {
                // the leader's MMAs read this CTA's stages: every use is
                // released before the CTA may exit
                for (int j = 0; j < C::S && !fail; ++j, ++it)
                    if (it >= (uint32_t)C::S && !umma::mbar_wait(&empty[it % C::S], ((it / C::S) & 1u) ^ 1u)) fail = true;
            }
            // no copy may still be landing in shared memory when the CTA exits
            // (the peer's copies complete on the leader's barriers)
            if (leader)
                for (uint32_t k = (it_end > (uint32_t)C::S ? it_end - C::S : 0u); k < it_end; ++k)
                    if (!umma::mbar_wait(&full[k % C::S], (k / C::S) & 1u, 200000000LL)) fail = true;
        }
    } else if (warp == 1) {
        // ----------------------------------------------- MMA issuer (leader)
        if (lane == 0 && leader) {
            constexpr int MM = PAIR ? 2 * BM : BM;
            constexpr uint32_t idesc = kMN ? umma::idesc_bf16_f32_mn(MM, BN) : umma::idesc_bf16_f32(MM, BN);
            auto commit = [&](uint64_t *bar) {
                if constexpr (PAIR) umma::mma_commit_pair_mc(bar, (uint16_t)0x3);
                else umma::mma_commit(bar);
            };
            const uint64_t da0 = kMN ? umma::sdesc_mnmajor_sw128(umma::smem_u32(smem), 8192)
                                     : umma::sdesc_kmajor_sw128(umma::smem_u32(smem));
            constexpr uint64_t kB = C::A_BYTES >> 4, kStage = C::STAGE >> 4, kStep = (kMN ? 2048 : 32) >> 4;
            uint32_t s = 0, ph = 0, j = 0;
            for (int t = t_first; t < total && !fail; t += t_step, ++j) {
                const int kb0 = t / per_split * a.kb_per_split;
                const int nkb = min(a.kb_per_split, kb_total - kb0);
                const uint32_t buf = j & 1u;
                if (j >= 2 && !umma::mbar_wait(&acc_empty[buf], ((j >> 1) & 1u) ^ 1u)) { fail = true; break; }
                umma::tc_fence_after();
                const uint32_t d_tmem = tmem + buf * BN;
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!umma::mbar_wait(&full[s], ph)) { fail = true; break; }
                    umma::tc_fence_after();
                    const uint64_t da = da0 + s * kStage;
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k) {
                        const uint32_t acc = (kb > 0 || k > 0) ? 1u : 0u;
                        if constexpr (PAIR) umma::mma_bf16_pair(d_tmem, da + k * kStep, da + (kB + k * kStep), idesc, acc);
                        else umma::mma_bf16(d_tmem, da + k * kStep, da + (kB + k * kStep), idesc, acc);
                    }
                    commit(&empty[s]);
                    if (++s == (uint32_t)C::S) { s = 0; ph ^= 1u; }
                }
                commit(&acc_full[buf]);
            }
            if constexpr (PAIR) {   // every MMA issued has completed before tensor memory is freed
                umma::mma_commit_pair_mc(drain, (uint16_t)0x1);
                if (!umma::mbar_wait(drain, 0u, 200000000LL)) fail = true;
            }
        }
    } else {
        // ------------------------------------------------ epilogue (each CTA)
        const int ew = warp - 2;
        const int q = warp & 3;                    // TMEM lane quarter this warp may access
        const int hcol = C::SPLIT_N ? (ew >> 2) * C::COLS : 0;   // this warp's first column
        const bool active = C::SPLIT_N || (ew < 4);
        const int row = q * 32 + lane;
        uint8_t *stg = stg_base + ew * 4096;
        if (EPI == kEpiHidden || EPI == kEpiOutPhys || EPI == kEpiOutLoss) {
            for (int col = threadIdx.x - 64; col < a.N; col += 32 * C::WARPS) sbias[col] = __ldg(a.bias + col);
            named_barrier_epi<32 * C::WARPS>();
        }
        GradBoxes gb;
        gb.full = gfull + 2 * ew;
        // (kEpiDx, lane 0) ask for the next GeLU'(z) box: box `nload` of this
        // warp's sequence, COLS / 32 a tile
        auto refill = [&]() {
            constexpr uint32_t G = C::COLS / 32 > 0 ? C::COLS / 32 : 1;
            const int t = t_first + (int)(gb.nload / G) * t_step;
            if (t >= total) return;
            int split, mt, n0;
            tile_of<BN, PAIR>(a, t, rank, split, mt, n0);
            umma::bulk_wait_read0();   // the store from this box has left
            uint64_t *bar = &gb.full[gb.nload & 1u];
            umma::mbar_arrive_expect_tx(bar, 2048);
            umma::tma_load_2d_hint(stg + (gb.nload & 1u) * 2048, &a.tm_gd, bar, n0 + hcol + (int)(gb.nload % G) * 32,
                                   mt * BM + q * 32, umma::l2_evict_first());
            ++gb.nload;
        };
        if (EPI == kEpiDx && lane == 0) refill();
        const uint32_t ae0 = PAIR ? umma::mapa_shared(umma::smem_u32(&acc_empty[0]), 0u) : 0u;
        const uint32_t ae1 = PAIR ? umma::mapa_shared(umma::smem_u32(&acc_empty[1]), 0u) : 0u;
        uint32_t j = 0;
        for (int t = t_first; t < total; t += t_step, ++j) {
            int split, mt, n0;
            tile_of<BN, PAIR>(a, t, rank, split, mt, n0);
            const bool tile_ok = mt < a.m_tiles;   // (an odd M-tile count leaves a pair's second CTA without)
            const int m0 = mt * BM;
            const int m = m0 + row;
            const bool mval = tile_ok && m < a.M;
            const uint32_t buf = j & 1u;
            if (EPI == kEpiDx && lane == 0 && !fail) refill();
            // after a timed-out wait this warp skips its work but keeps taking
            // part in the named barriers, so the other epilogue warps finish
            if (!fail && !umma::mbar_wait(&acc_full[buf], (j >> 1) & 1u)) fail = true;
            fail = __any_sync(0xffffffffu, fail);   // warp-uniform: tcgen05.ld needs the whole warp
            umma::tc_fence_after();
            const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + buf * BN + hcol;
            float *rd = red + buf * C::RED_FLOATS;   // this tile's; the other one may still be read
            float lsum = epilogue_tile<BN, EPI>(a, taddr, m, mval, n0, hcol, q, lane, split, rd, sbias, active, tile_ok,
                                                fail, stg, m0, gb, refill);
            // the accumulator buffer may be reused once every warp has read it
            umma::tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if constexpr (PAIR) umma::mbar_arrive_cluster(buf ? ae1 : ae0);
                else umma::mbar_arrive(&acc_empty[buf]);
            }
            if (EPI == kEpiOutLoss || EPI == kEpiDx) {
                if (EPI == kEpiOutLoss) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
                    if (lane == 0 && active) rd[4 * BN + q] = lsum;
                }
                named_barrier_epi<32 * C::WARPS>();   // (one per tile: `rd` is written again two tiles on, behind the next one)
                const int tt = tile_ok ? threadIdx.x - 64 : BN;
                for (int col = tt; col < BN; col += 32 * C::WARPS)
                    a.colsum[(int64_t)mt * a.N + n0 + col] =
                        rd[col] + rd[BN + col] + rd[2 * BN + col] + rd[3 * BN + col];
                if (EPI == kEpiOutLoss && tile_ok && tt == 0)
                    a.loss_part[mt] = rd[4 * BN] + rd[4 * BN + 1] + rd[4 * BN + 2] + rd[4 * BN + 3];
            }
        }
        if (lane == 0) {
            // no box may still be landing, and staged stores complete, before shared memory goes
            if (EPI == kEpiDx)
                for (; gb.nuse < gb.nload; ++gb.nuse)
                    if (!umma::mbar_wait(&gb.full[gb.nuse & 1u], (gb.nuse >> 1) & 1u, 200000000LL)) fail = true;
            umma::bulk_wait0();
        }
    }
    __syncwarp();   // reconverge each warp (role lanes vs idle lanes) before the CTA barrier
    if (fail) atomicExch(a.err, 1);
    umma::tc_fence_before();
    __syncthreads();
    // a pair's MMAs, barrier signals and remote arrivals are all done before
    // either CTA frees its tensor memory or exits
    if constexpr (PAIR) umma::cluster_sync();
    if (warp == 1) {
        __syncwarp();
        umma::tc_fence_after();
        if constexpr (PAIR) umma::tmem_dealloc_pair(tmem, C::TMEM_COLS);
        else umma::tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

}  // namespace mlp
