// Inference of the whole surrogate MLP with the activations resident in
// shared memory: a CTA pair (cta_group::2 MMAs, M = 256) takes a block of 256
// rows through every layer before it moves to its next block, each CTA keeping
// its 128 rows' activation (128 x W BF16, in the 128-byte-swizzled K-major
// layout the MMA reads) in its own shared memory.  Only the weights stream
// from L2, each CTA loading its half of every N-tile (the pair MMA's B split
// along N), so the L2 traffic is the weights once per 256 rows and nothing
// else: no activation leaves the SM, and no CTA waits on another pair.
//
// Each hidden layer's output (N = W) is computed as two N-tiles of BN = W / 2
// columns, accumulated in tensor memory at columns [0, BN) and [BN, 2 BN)
// (all 512 columns for W = 512).  The activation lies in slots of one K-block
// (64 columns), W / 64 + 1 of them: a layer reads its input from W / 64 slots
// and writes the first K-block of its output to the spare one, the next ones
// to slots whose K-block its own second N-tile has read by then, so the slots
// rotate by one from layer to layer.  In MMA order:
//   N-tile 0 of layer l (all K)        -> its epilogue starts at once: K-block 0
//                                         of the output into the spare slot,
//   N-tile 1, K-blocks 0 .. nc - 2     -> its other K-blocks (nc = W / 128 in
//                                         all) into the slots just read,
//   N-tile 1, the rest                 -> the epilogue of N-tile 1, reported in
//                                         two halves,
//   N-tile 0 of layer l + 1: K-blocks 0 .. nc - 1 (written long before), then
//   the two halves as they arrive.
// With W / 64 slots (the output written over the input in halves, the first
// epilogue waiting for half of N-tile 1) the MMAs and the epilogues alternated
// more than they overlapped (4 Mi rows, width 512, four hidden layers, the
// whole call: 5.64 ms; with the spare slot 5.39 ms).  What holds it now: the
// issuing thread, which shares its scheduler with four epilogue warps, takes
// ~680 cycles per K-block of 512 cycles of tensor work (73 % of the time), and
// at a block's boundary the input layer's epilogue waits for the output layer
// (14 %); weight stages 7 %.
// The input layer (the standardised inputs as a TMA tile of 32 columns in a
// buffer of their own) and the output layer (N = 16, accumulated in the first
// 16 columns of the second accumulator, which the last epilogue's first half
// has read) are interleaved with the neighbouring row blocks:
//   input N-tile 0 of block r, output layer of block r - 1, input N-tile 1 of
//   block r, hidden layers of block r, ...
// Barriers: a stage ring (full / empty) and the input buffer (x_full /
// x_empty) between the TMA producers and the MMA issuer; MMA completion
// (tcgen05.commit, multicast to both CTAs) tells the epilogues that N-tile 0
// or 1 is ready (`hid`), that the slots of N-tile 0's later K-blocks are no
// longer read (`slots`), or that the output layer is done (`outf`); one
// arrival per CTA on the leader's barriers, after a named barrier of that
// CTA's epilogue warps, tells the MMA issuer that N-tile 0's columns are
// written and its accumulator read (`epi0`), that the first and the second
// half of N-tile 1's are (`epi1`), or that the output accumulator has been
// read (`out_done`).  The issuing thread does as little as possible between
// MMAs (the tensor core does not queue far ahead of it): indices and phases
// advance by increments and shared-memory descriptors by 64-bit adds.
// Every wait is bounded; a failed wait sets the error flag, and every role
// then stops, lets its copies and MMAs in flight complete, and returns (the
// epilogue warps keep their trip counts, so their named barriers always
// complete).
#pragma once

#include "mlp_gemm.cuh"

namespace mlp {

constexpr int kResEpiWarps = 16;                       // four per TMEM lane quarter
constexpr int kResThreads = 64 + 32 * kResEpiWarps;    // producer, MMA issuer, epilogue
constexpr int kResOutBN = 16;                          // padded output width
constexpr int kResXCols = 32;                          // input columns: the standardised inputs' hi and lo parts

struct ResidentArgs {
    CUtensorMap tm_x;                     // standardised inputs [rows][64], box 32 x 128 (64-byte swizzle)
    CUtensorMap tm_w[kFusedMaxLayers];    // W_l [out][in]: box 64 x (W / 4) (hidden, this CTA's half of
                                          // an N-tile), 64 x 8 (output layer)
    const float *bias[kFusedMaxLayers];   // b_l [out_pad]
    int M;                                // rows of the chunk
    int L;                                // hidden layers
    int W;                                // width: 256 or 512
    float *out6;                          // [nout][ld6] physical outputs of the chunk's rows
    long long ld6;
    const float *out_mean, *out_std;      // [nout] de-standardisation
    int nout;                             // outputs in use (<= 16)
    const float *add_h;                   // per-row term added to output 2 (h), or NULL
    int log_mask;                         // bit j set = output j was learned as its logarithm
    int *err;                             // set to 1 when a bounded wait runs out
    long long wait_cycles;                // limit of every bounded wait
    int stall_test;                       // test hook: the MMA issuer waits for one epilogue too many
};

// Shared memory: the activation's slots (128 rows x 64 BF16 each), the stage
// ring, the input tile (128 x 32 BF16), the barriers, the biases of every layer.
struct ResCfg {
    static constexpr int kMaxSmem = 232448;   // 227 KB opt-in per CTA
    static constexpr int STAGE = 16384;       // this CTA's half of a weight K-block (at most 128 x 64 BF16)
    static constexpr int SLOT = 16384;        // 128 x 64 BF16
    static constexpr int XBYTES = 128 * kResXCols * 2;
    static constexpr int BAR_BYTES = 256;
    __host__ __device__ static int slots(int W) { return W / 64 + 1; }
    __host__ __device__ static int bias_bytes(int L, int W) { return (L * W + kResOutBN) * 4; }
    __host__ __device__ static int smem_bytes(int L, int W, int stages)
    {
        return 1024 + slots(W) * SLOT + stages * STAGE + XBYTES + BAR_BYTES + bias_bytes(L, W);
    }
    // weight stages: four, or three where the biases of a deep network leave
    // no room (width 512, five layers and more)
    static int stages(int L, int W) { return smem_bytes(L, W, 4) <= kMaxSmem ? 4 : 3; }
    // widths this kernel takes: two N-tiles of W / 2 columns fill at most the
    // 512 TMEM columns
    static bool supports(int L, int W)
    {
        return (W == 256 || W == 512) && L >= 1 && L < kFusedMaxLayers && smem_bytes(L, W, stages(L, W)) <= kMaxSmem;
    }
};

// Position in the stage ring: index and phase parity, advanced by increments
template <int S>
struct RingPos {
    uint32_t s = 0, ph = 0;
    __device__ __forceinline__ void next()
    {
        if (++s == (uint32_t)S) {
            s = 0;
            ph ^= 1u;
        }
    }
};

// Named barrier among `threads` threads (id 1..15; id 0 is __syncthreads)
__device__ __forceinline__ void named_sync(uint32_t id, uint32_t threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// GeLU(acc + b) of 16 accumulator columns, as BF16 into a slot of the resident
// activation (128 rows x 128 B, 16-byte chunks swizzled by the row's index
// within its 8-row atom, as TMA's 128-byte swizzle places them): the two
// chunks at shared addresses d0 and d1.
__device__ __forceinline__ void act_chunk(const uint32_t (&r)[16], const float *sb, uint32_t d0, uint32_t d1)
{
    const float4 *b4 = reinterpret_cast<const float4 *>(sb);
    uint32_t pk[8];
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) {
        const float4 b = b4[jj];
        const float2 g0 = gelu2(make_float2(__uint_as_float(r[4 * jj]), __uint_as_float(r[4 * jj + 1])),
                                make_float2(b.x, b.y));
        const float2 g1 = gelu2(make_float2(__uint_as_float(r[4 * jj + 2]), __uint_as_float(r[4 * jj + 3])),
                                make_float2(b.z, b.w));
        pk[2 * jj] = pack_bf16(g0.x, g0.y);
        pk[2 * jj + 1] = pack_bf16(g1.x, g1.y);
    }
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(d0), "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3])
                 : "memory");
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(d1), "r"(pk[4]), "r"(pk[5]), "r"(pk[6]), "r"(pk[7])
                 : "memory");
}

// The slot after `s` (by n) in the rotation
template <int NSLOT>
__device__ __forceinline__ uint32_t slot_add(uint32_t s, uint32_t n)
{
    const uint32_t t = s + n;
    return t >= (uint32_t)NSLOT ? t - (uint32_t)NSLOT : t;
}

template <int W, int S>
__global__ void __launch_bounds__(kResThreads, 1) mlp_resident_kernel(const __grid_constant__ ResidentArgs a)
{
    static_assert(W == 256 || W == 512, "resident activations: width 256 or 512");
    constexpr int BN = W / 2, nkb = W / 64, nc = nkb / 2, NSLOT = nkb + 1;
    constexpr uint32_t kStageDesc = ResCfg::STAGE >> 4;   // descriptor address units per stage or slot
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int L = a.L;
    uint8_t *act = smem;
    uint8_t *stage = smem + NSLOT * ResCfg::SLOT;
    uint8_t *xbuf = stage + S * ResCfg::STAGE;
    uint64_t *full = reinterpret_cast<uint64_t *>(xbuf + ResCfg::XBYTES);
    uint64_t *empty = full + S;
    uint64_t *x_full = empty + S;     // input tile landed (both CTAs')
    uint64_t *x_empty = x_full + 1;   // input tile no longer read
    uint64_t *hid = x_empty + 1;      // [2] N-tile b ready
    uint64_t *slots = hid + 2;        // the slots of N-tile 0's K-blocks 1 .. nc - 1 no longer read
    uint64_t *outf = slots + 1;       // output layer done
    uint64_t *epi0 = outf + 1;        // (leader) N-tile 0's columns written, accumulator 0 read
    uint64_t *epi1 = epi0 + 1;        // [2] (leader) the halves of N-tile 1's columns written and read
    uint64_t *out_done = epi1 + 2;    // (leader) output accumulator read
    uint64_t *drain = out_done + 1;   // (leader) every MMA issued has completed
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    float *sbias = reinterpret_cast<float *>(reinterpret_cast<uint8_t *>(full) + ResCfg::BAR_BYTES);   // [L W + 16]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = umma::cluster_ctarank();
    const bool leader = rank == 0;
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    const int R = (a.M + 255) / 256;                                  // row blocks of 256
    const int nr = pair < R ? (R - pair + npairs - 1) / npairs : 0;   // this pair's row blocks
    const long long wc = a.wait_cycles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            umma::mbar_init(&full[s], 1);
            umma::mbar_init(&empty[s], 1);
        }
        umma::mbar_init(x_full, 1);
        umma::mbar_init(x_empty, 1);
        umma::mbar_init(&hid[0], 1);
        umma::mbar_init(&hid[1], 1);
        umma::mbar_init(slots, 1);
        umma::mbar_init(outf, 1);
        umma::mbar_init(epi0, 2);
        umma::mbar_init(&epi1[0], 2);
        umma::mbar_init(&epi1[1], 2);
        umma::mbar_init(out_done, 2);
        umma::mbar_init(drain, 1);
        *tmem_slot = 0u;
        umma::fence_mbar_init();
        umma::tma_prefetch_desc(&a.tm_x);
    }
    __syncthreads();
    if (warp == 1) {
        umma::tmem_alloc_pair(tmem_slot, 512);
        umma::tmem_relinquish_pair();
    }
    for (int e = threadIdx.x; e < L * W + kResOutBN; e += blockDim.x) {
        const int l = (e < L * W) ? e / W : L;
        const int n = (e < L * W) ? e - l * W : e - L * W;
        sbias[e] = __ldg(a.bias[l] + n);
    }
    umma::tc_fence_before();
    __syncthreads();
    umma::cluster_sync();   // both CTAs' barriers initialised before any copy or MMA signals them
    // the kernel before this one writes the inputs (the biases above are older
    // than its start: it is launched in stream order)
    umma::pdl_wait();
    umma::pdl_release();
    umma::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    bool fail = false;

    if (warp == 0) {
        // ------------------------------------------------ TMA producer (each CTA)
        if (lane == 0) {
            RingPos<S> rp;
            uint32_t it = 0, nx = 0;
            const uint32_t wbytes = 2u * (uint32_t)(BN / 2) * 128u;   // the pair's halves of a weight K-block
            const int hrow = (int)rank * (BN / 2);                       // this CTA's rows of an N-tile
            // the next stage, once free; false after a failed wait
            auto next_stage = [&](uint32_t bytes) -> bool {
                if (fail) return false;
                if (it >= (uint32_t)S && !umma::mbar_wait(&empty[rp.s], rp.ph ^ 1u, wc)) {
                    fail = true;
                    return false;
                }
                if (leader) umma::mbar_arrive_expect_tx(&full[rp.s], bytes);
                return true;
            };
            auto put = [&](const CUtensorMap *tm, int c0, int c1) {
                if (!next_stage(wbytes)) return;
                umma::tma_load_2d_pair(stage + rp.s * ResCfg::STAGE, tm, umma::mapa_shared(umma::smem_u32(&full[rp.s]), 0u),
                                       c0, c1);
                ++it;
                rp.next();
            };
            // the output layer's weights, this CTA's 8 rows of every K-block, in one stage
            auto put_out = [&]() {
                if (!next_stage(2u * (uint32_t)nkb * 1024u)) return;
                const uint32_t bar = umma::mapa_shared(umma::smem_u32(&full[rp.s]), 0u);
                for (int k = 0; k < nkb; ++k)
                    umma::tma_load_2d_pair(stage + rp.s * ResCfg::STAGE + k * 1024, &a.tm_w[L], bar, k * 64, (int)rank * 8);
                ++it;
                rp.next();
            };
            for (int i = 0; i < nr && !fail; ++i) {
                const int r = pair + i * npairs;
                // the input tile, once the previous block's input layer has read it
                if (i > 0 && !umma::mbar_wait(x_empty, (uint32_t)(i - 1) & 1u, wc)) {
                    fail = true;
                    break;
                }
                if (leader) umma::mbar_arrive_expect_tx(x_full, 2u * (uint32_t)ResCfg::XBYTES);
                umma::tma_load_2d_pair(xbuf, &a.tm_x, umma::mapa_shared(umma::smem_u32(x_full), 0u), 0,
                                       r * 256 + (int)rank * 128);
                ++nx;
                put(&a.tm_w[0], 0, hrow);
                if (i > 0) put_out();
                put(&a.tm_w[0], 0, BN + hrow);
                for (int l = 1; l < L; ++l)
                    for (int b = 0; b < 2; ++b)
                        for (int k = 0; k < nkb; ++k) put(&a.tm_w[l], k * 64, b * BN + hrow);
            }
            if (nr > 0) put_out();
            const uint32_t it_end = it;
            // the leader's MMAs read this CTA's stages: every use is released
            // before the CTA may exit
            for (int j = 0; j < S && !fail; ++j) {
                if (it >= (uint32_t)S && !umma::mbar_wait(&empty[rp.s], rp.ph ^ 1u, wc)) fail = true;
                ++it;
                rp.next();
            }
            // no copy may still be landing in shared memory at exit (the
            // peer's copies complete on the leader's barriers)
            if (leader) {
                for (uint32_t k = (it_end > (uint32_t)S ? it_end - S : 0u); k < it_end; ++k)
                    if (!umma::mbar_wait(&full[k % S], (k / S) & 1u, 200000000LL)) fail = true;
                if (nx > 0 && !umma::mbar_wait(x_full, (uint32_t)(nx - 1) & 1u, 200000000LL)) fail = true;
            }
            if (fail) atomicExch(a.err, 1);
        }
    } else if (warp == 1) {
        // ----------------------------------------------- MMA issuer (leader)
        if (lane == 0 && leader) {
            RingPos<S> rp;
            uint32_t ne0 = 0, ne1a = 0, ne1b = 0, no = 0, nxf = 0;
            const uint32_t id_h = umma::idesc_bf16_f32(256, BN), id_o = umma::idesc_bf16_f32(256, kResOutBN);
            const uint32_t acc0 = tmem, acc1 = tmem + (uint32_t)BN;
            const uint64_t d_act = umma::sdesc_kmajor_sw128(umma::smem_u32(act));
            const uint64_t d_x = umma::sdesc_kmajor_sw64(umma::smem_u32(xbuf));
            const uint64_t d_st = umma::sdesc_kmajor_sw128(umma::smem_u32(stage));
            uint32_t sl = 0;   // the slot of the current activation's K-block 0
            auto wait_bar = [&](uint64_t *bar, uint32_t &n) {
                if (!fail && !umma::mbar_wait(bar, n & 1u, wc)) fail = true;
                ++n;
                umma::tc_fence_after();
            };
            // the next stage, once landed: its descriptor
            auto take = [&]() -> uint64_t {
                if (!fail && !umma::mbar_wait(&full[rp.s], rp.ph, wc)) fail = true;
                umma::tc_fence_after();
                return d_st + (uint64_t)(rp.s * kStageDesc);
            };
            // release the stage just read, once the MMAs reading it complete
            auto give = [&]() {
                umma::mma_commit_pair_mc(&empty[rp.s], (uint16_t)0x3);
                rp.next();
            };
            // one K-block: four K = 16 MMAs (descriptor address +32 B each)
            auto kblock = [&](uint32_t d, uint64_t da, uint64_t db, uint32_t id, bool acc_in) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    umma::mma_bf16_pair(d, da + 2 * kk, db + 2 * kk, id, (acc_in || kk > 0) ? 1u : 0u);
            };
            // an N-tile of the input layer: K = 32
            auto input_tile = [&](uint32_t d) {
                const uint64_t db = take();
                if (fail) return;
#pragma unroll
                for (int kk = 0; kk < kResXCols / 16; ++kk)
                    umma::mma_bf16_pair(d, d_x + 2 * kk, db + 2 * kk, id_h, kk > 0 ? 1u : 0u);
                give();
            };
            // the output layer (epi0 waited before); with `next`, the slots it
            // has read are reported to the next block's first epilogue
            auto output_layer = [&](bool next) {
                wait_bar(&epi1[0], ne1a);   // and the columns it accumulates in have been read
                const uint64_t db = take();
                uint32_t s = sl;
                for (int k = 0; k < nkb && !fail; ++k) {
                    if (k == nc + nc / 2) wait_bar(&epi1[1], ne1b);
                    if (fail) break;
                    kblock(acc1, d_act + (uint64_t)(s * kStageDesc), db + (uint64_t)(k * 64), id_o, k > 0);
                    s = slot_add<NSLOT>(s, 1u);
                    if (next && k == nc - 2) umma::mma_commit_pair_mc(slots, (uint16_t)0x3);
                }
                if (fail) return;
                give();
                umma::mma_commit_pair_mc(outf, (uint16_t)0x3);
            };
            for (int i = 0; i < nr && !fail; ++i) {
                if (i > 0) wait_bar(epi0, ne0);   // accumulator 0 read by the last layer's epilogue
                wait_bar(x_full, nxf);
                input_tile(acc0);
                if (fail) break;
                umma::mma_commit_pair_mc(&hid[0], (uint16_t)0x3);
                if (i > 0)
                    output_layer(true);   // of the previous row block
                else
                    umma::mma_commit_pair_mc(slots, (uint16_t)0x3);
                if (fail) break;
                if (i > 0) wait_bar(out_done, no);
                input_tile(acc1);
                if (fail) break;
                umma::mma_commit_pair_mc(x_empty, (uint16_t)0x3);
                umma::mma_commit_pair_mc(&hid[1], (uint16_t)0x3);
                sl = slot_add<NSLOT>(sl, (uint32_t)NSLOT - 1u);
                for (int l = 1; l < L && !fail; ++l) {
                    uint32_t s = sl;
                    for (int k = 0; k < nkb && !fail; ++k) {
                        if (k == 0) {
                            wait_bar(epi0, ne0);
                            if (a.stall_test && i == 0 && l == 1) wait_bar(epi0, ne0);   // never arrives
                        }
                        if (k == nc) wait_bar(&epi1[0], ne1a);
                        if (k == nc + nc / 2) wait_bar(&epi1[1], ne1b);
                        const uint64_t db = take();
                        if (fail) break;
                        kblock(acc0, d_act + (uint64_t)(s * kStageDesc), db, id_h, k > 0);
                        s = slot_add<NSLOT>(s, 1u);
                        give();
                    }
                    if (fail) break;
                    umma::mma_commit_pair_mc(&hid[0], (uint16_t)0x3);
                    s = sl;
                    for (int k = 0; k < nkb && !fail; ++k) {
                        const uint64_t db = take();
                        if (fail) break;
                        kblock(acc1, d_act + (uint64_t)(s * kStageDesc), db, id_h, k > 0);
                        s = slot_add<NSLOT>(s, 1u);
                        give();
                        if (k == nc - 2) umma::mma_commit_pair_mc(slots, (uint16_t)0x3);
                    }
                    if (!fail) umma::mma_commit_pair_mc(&hid[1], (uint16_t)0x3);
                    sl = slot_add<NSLOT>(sl, (uint32_t)NSLOT - 1u);
                }
            }
            if (nr > 0 && !fail) {
                wait_bar(epi0, ne0);
                output_layer(false);
            }
            // every MMA issued has completed before tensor memory is freed
            umma::mma_commit_pair_mc(drain, (uint16_t)0x1);
            if (!umma::mbar_wait(drain, 0u, 200000000LL)) fail = true;
            if (fail) atomicExch(a.err, 1);
        }
    } else {
        // ------------------------------------------------ epilogue (each CTA)
        const int ew = warp - 2;        // 0..15
        const int q = warp & 3;         // TMEM lane quarter this warp may access
        const int cg = ew >> 2;         // 16-column quarter of a K-block
        const int row = q * 32 + lane;  // this thread's row of the CTA's 128
        const uint32_t lanes = (uint32_t)(q * 32) << 16;
        const uint32_t act_row = umma::smem_u32(act) + (uint32_t)(row * 128);
        // this thread's two 16-byte chunks of a slot's row, swizzled by row % 8
        const uint32_t d0 = act_row + (uint32_t)(((row & 7) ^ (2 * cg)) << 4);
        const uint32_t d1 = act_row + (uint32_t)(((row & 7) ^ (2 * cg + 1)) << 4);
        const uint32_t epi0_c = umma::mapa_shared(umma::smem_u32(epi0), 0u);
        const uint32_t epi1a_c = umma::mapa_shared(umma::smem_u32(&epi1[0]), 0u);
        const uint32_t epi1b_c = umma::mapa_shared(umma::smem_u32(&epi1[1]), 0u);
        const uint32_t out_c = umma::mapa_shared(umma::smem_u32(out_done), 0u);
        uint32_t nh0 = 0u, nh1 = 0u, nsl = 0u, nof = 0u;
        uint32_t sl = 0;   // the slot of the current layer's input K-block 0
        // failed waits are not retried, but the trip counts stay the same, so
        // every named barrier completes
        auto wait_bar = [&](uint64_t *bar, uint32_t &n) {
            if (!fail && !umma::mbar_wait(bar, n & 1u, wc)) fail = true;
            ++n;
            fail = __any_sync(0xffffffffu, fail);   // warp-uniform: tcgen05.ld needs the whole warp
            umma::tc_fence_after();
        };
        // this warp's part of what it wrote and read is done: report it
        auto report = [&](uint32_t bar_c) {
            umma::fence_async_smem();   // the activation writes, visible to the tensor core
            umma::tc_fence_before();
            named_sync(1, 32 * kResEpiWarps);
            if (ew == 0 && lane == 0 && !fail) umma::mbar_arrive_cluster(bar_c);
        };
        // warps 2..5 (one per lane quarter): de-standardised outputs of row block r
        // (the per-row term and the first 8 outputs' bias, scale and shift are
        // loaded before the wait; the rest is read after it)
        auto output_epilogue = [&](int r, bool signal) {
            const int m = r * 256 + (int)rank * 128 + row;
            const float hadd = (a.add_h && m < a.M) ? __ldg(a.add_h + m) : 0.f;
            const float *sb = sbias + L * W;
            float ob[8], os[8], om[8];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
                ob[jj] = sb[jj];
                os[jj] = __ldg(a.out_std + jj);
                om[jj] = __ldg(a.out_mean + jj);
            }
            wait_bar(outf, nof);
            if (!fail) {
                uint32_t rr[16];
                umma::tmem_ld16(tmem + lanes + (uint32_t)BN, rr);
                umma::tmem_ld_wait(rr);
                if (m < a.M) {
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj) {
                        if (jj >= a.nout) break;
                        float qv = jj < 8 ? (__uint_as_float(rr[jj]) + ob[jj & 7]) * os[jj & 7] + om[jj & 7]
                                          : (__uint_as_float(rr[jj]) + sb[jj]) * __ldg(a.out_std + jj) +
                                                __ldg(a.out_mean + jj);
                        if (jj == 2) qv += hadd;
                        a.out6[(long long)jj * a.ld6 + m] = ((a.log_mask >> jj) & 1) ? __expf(qv) : qv;
                    }
                }
            }
            umma::tc_fence_before();
            named_sync(2, 128);
            if (signal && ew == 0 && lane == 0 && !fail) umma::mbar_arrive_cluster(out_c);
        };
        for (int i = 0; i < nr; ++i) {
            if (i > 0 && ew < 4) output_epilogue(pair + (i - 1) * npairs, true);
            for (int l = 0; l < L; ++l) {
                // output K-block c goes to slot sl + c - 1 (c = 0: the spare one)
                uint32_t so = slot_add<NSLOT>(sl, (uint32_t)NSLOT - 1u);
                const float *sb = sbias + l * W + cg * 16;
                uint32_t ta = tmem + lanes + (uint32_t)(cg * 16);
                uint32_t r[2][16];
                // one K-block of an N-tile's columns after the other: the next
                // one's accumulator is loaded while this one's GeLU runs, except
                // across a wait or a report, which no load in flight spans
#pragma unroll
                for (int c = 0; c < nkb; ++c) {
                    const bool fresh = c == 0 || c == 1 || c == nc || c == nc + nc / 2;   // after a wait or a report
                    if (c == 0) wait_bar(&hid[0], nh0);
                    if (c == 1) wait_bar(slots, nsl);
                    if (c == nc) wait_bar(&hid[1], nh1);
                    if (!fail) {
                        if (fresh) umma::tmem_ld16(ta + (uint32_t)(c * 64), r[c & 1]);
                        umma::tmem_ld_wait(r[c & 1]);
                        const int n = c + 1;
                        if (n != 1 && n != nc && n != nc + nc / 2 && n != nkb)
                            umma::tmem_ld16(ta + (uint32_t)(n * 64), r[n & 1]);
                        act_chunk(r[c & 1], sb + c * 64, d0 + so * (uint32_t)ResCfg::SLOT, d1 + so * (uint32_t)ResCfg::SLOT);
                    }
                    so = slot_add<NSLOT>(so, 1u);
                    if (c == nc - 1) report(epi0_c);
                    if (c == nc + nc / 2 - 1) report(epi1a_c);
                    if (c == nkb - 1) report(epi1b_c);
                }
                sl = slot_add<NSLOT>(sl, (uint32_t)NSLOT - 1u);
            }
        }
        if (nr > 0 && ew < 4) output_epilogue(pair + (nr - 1) * npairs, false);
        if (fail && lane == 0) atomicExch(a.err, 1);
    }
    __syncwarp();
    umma::tc_fence_before();
    __syncthreads();
    // the pair's MMAs, barrier signals and remote arrivals are all done before
    // either CTA frees its tensor memory or exits
    umma::cluster_sync();
    if (warp == 1) {
        __syncwarp();
        umma::tc_fence_after();
        umma::tmem_dealloc_pair(tmem, 512);
    }
}

}  // namespace mlp
