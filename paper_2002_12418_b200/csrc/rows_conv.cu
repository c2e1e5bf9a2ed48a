// Stride-1 convolution in one kernel: input transform, tensor-core product and output transform, one axis at a time (rows_plan.h).
//
// A work item is 128 * MT cells x bn output channels.  The producer warps read x, apply B^T along the row (nothing where m = 1),
// split the values into BF16 hi + lo and write them, 16 channels per stage, as K-major rows of 32 bytes in the 32-byte swizzle:
// per operand plane (transform position) and half, `rows` consecutive cells.  The swizzle depends on the address alone, so
// kernel row a is the same plane read a * Wq rows further on: an element of x is converted once per item and serves every
// kernel row.  One warp streams the weights, stored at preparation time in the byte order of their shared-memory tiles, with bulk
// copies; one issues tcgen05.mma: hi*hi + lo*hi + hi*lo for every (kernel row, position) into one accumulator per position.
// Eight warps read the accumulators, apply A^T, bias and ReLU and store y.  Neither V nor M exists in memory.
//
// What bounds it: no memory level is near its rate (256 channels 56 x 56 BF16: tensor pipe 45 % busy, shared-memory banks 37 %, L2 24 %,
// DRAM 10 %).  An instruction of 128 x N x 16 alone takes max(N / 2, 57 + N / 7) cycles, so narrow channel blocks cost as much as 96
// channels.  With clocks in each role, which slow it by themselves, the issuing warp spent 112 cycles an instruction at N = 128
// and 168 at N = 256 (75 and 128 alone) and 630 to 660 a stage waiting; why they are longer there was not separated.  Measured, one kernel against what ran
// before: one image 64 channels 56 x 56 13.1 -> 8.5 us, 128 channels 28 x 28 12.2 -> 8.6, batch 32 64 channels 51 -> 28 (m = 2),
// 128 channels 31 -> 23 (m = 2), 7 images 100 -> 72 channels 35 x 45 18.8 -> 13.6, 192 channels 17 x 17 1 x 7 batch 32 28.8 -> 21.7,
// 256 channels 56 x 56 batch 64 BF16 249 -> 218.  Error against 64 bits with hi + lo operands, 160 random layers: 4 to 7e-6 (m = 1; to 6e-5 at
// 30000 terms, by the accumulator's own rounding, where two-dimensional Winograd had 1.7e-4) and 7e-6 at most (m = 2).  One BF16 product:
// 2.0 to 2.6e-3, that of the BF16 products it replaced, 0.33 to 0.90 of F(2, 5), F(2, 7), F(6, 3) and F(4, 5) on one TF32 product, and of F(4, 3)
// 0.75 for inputs around zero and 0.92 behind a ReLU in the mean of 116 layers, five of them 1.03 to 1.06, one 1.25.
//
// SPLIT: a cluster of p.split CTAs takes one item, each CTA a share of the input channels; the partial outputs (after A^T, which
// is linear) meet in distributed shared memory.
#include "rows_conv.h"

#include <cuda_bf16.h>

#include "cluster.cuh"
#include "umma.cuh"

namespace mnnb {

namespace {

// Two outputs per cell keep the operands of one task in flight in twelve producer warps, the definition of three tasks in ten: what the
// registers of a block allow (64 channels 56 x 56 batch 32, two outputs: 42 us with ten warps and two tasks, 35 with ten and one, 28
// with twelve to sixteen and one).  Eight epilogue warps, as four spend 140 cycles per store on short K loops (definition 37 -> 30 us).
constexpr int kEpiWarps = 8;
constexpr int kFirstEpi = 2, kFirstProducer = kFirstEpi + kEpiWarps;
template <int M>
constexpr int kProducers = M == 1 ? 10 : 12;
template <int M>
constexpr int kRowsThreads = 32 * (kFirstProducer + kProducers<M>);
constexpr int kMaxSharedBias = 2048;
constexpr int kErrRowsStream = 61, kErrRowsMmaA = 62, kErrRowsMmaB = 63, kErrRowsMmaAcc = 64, kErrRowsEpilogue = 65, kErrRowsProducer = 66;

struct RowsParams {
    const float* x;
    const float* bias;
    float* y;
    const uint8_t* U;
    int* status;
    unsigned T, n_items, n_tile_blocks;
    int Cin, Cout, H, W, OH, OW, steps, step_rows, tap_rows, taps_down, pad_h, pad_w, Hq, Wq, rows, rows_pad, k_slots, bn, a_slots, b_slots, acc_bufs, tmem_cols, split, relu;
    float Bt[kRowsMaxAlpha * kRowsMaxAlpha], At[2 * kRowsMaxAlpha];
};

// High word of the shared-memory descriptors: 8-row groups 256 bytes apart, version, 32-byte swizzle.
constexpr uint32_t kDescHi = (256u >> 4) | (1u << 14) | (6u << 29);

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ bool is_number(float v) { return fabsf(v) <= 3.402823466e+38f; }

// max(v, 0) that keeps what is no number.
__device__ __forceinline__ float relu_nan(float v)
{
    float r;
    asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float2 add_pair(float2 a, float2 b)
{
    float2 r;
    asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

// Outputs of one cell that were stored as no finite number, again: the definition's sum in fp32 from x and the two halves of the
// stored weights.  For an infinite x, or a finite one that BF16 rounds to infinity, lo = x - hi is no number, and hi * hi may pass the
// largest number where the sum does not.  Columns col0, col0 + step, ... of channel block nb, which starts at channel co0.
// Behind the loop over items, a sum of its outputs tells a thread whether there are any: asked and answered inside the loop it cost
// finite layers 1 to 6 %, so nothing that shows (7 images 100 -> 72 channels 35 x 45 13.96 us without, 13.79 with, 14.2 inside; 29 images
// 32 -> 480 channels 96 x 20 44.2, 43.5 and 47.2).
template <int TAPS>
__device__ __noinline__ void rows_redo(const RowsParams& p, unsigned img, int i, int j, unsigned nb, int co0, int col0, int col1, int step)
{
    const size_t tile = (size_t)p.bn * 32, plane = (size_t)p.H * p.W;
    for (int col = col0; col < col1; col += step) {
        float* const at = p.y + (((size_t)img * p.Cout + co0 + col) * p.OH + i) * p.OW + j;
        if (is_number(*at)) continue;
        const float* xc = p.x + (size_t)img * p.Cin * plane;
        float s = 0.0f;
        for (int ci = 0; ci < p.Cin && s == s; ++ci, xc += plane) {
            const int c = ci & (kRowsChannels - 1);
            const uint8_t* u = p.U + ((size_t)nb * p.k_slots + ci / kRowsChannels) * p.steps * (TAPS * 2 * tile) + col * 32 + (((c >> 3) ^ ((col >> 2) & 1)) << 4) + (c & 7) * 2;
            for (int v = 0; v < p.steps; ++v)
                for (int t = 0; t < TAPS; ++t, u += 2 * tile) {
                    const int ih = i - p.pad_h + v + (p.taps_down ? t : 0), iw = j - p.pad_w + (p.taps_down ? 0 : t);
                    if (ih < 0 || ih >= p.H || iw < 0 || iw >= p.W) continue;
                    const float w = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(u)) + __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(u + tile));
                    s = fmaf(w, __ldg(xc + (size_t)ih * p.W + iw), s);
                }
        }
        s += p.bias ? __ldg(p.bias + co0 + col) : 0.0f;
        *at = p.relu ? fmaxf(s, 0.0f) : s;
    }
}

// M outputs per cell, KW taps along the row; MT tiles of 128 cells per item.  MODE: 1 one product of BF16 operands; 3 the three
// products of hi + lo operands; 2 the same three as two instructions, A_hi x [B_hi; B_lo] into two accumulators side by side
// and A_lo x B_hi into the first: an instruction spends 57 cycles on its left operand whatever its width.
template <int M, int KW, int MT, int MODE, bool SPLIT>
__global__ void __launch_bounds__(kRowsThreads<M>, 1) rows_conv_kernel(const __grid_constant__ RowsParams p)
{
    constexpr int ALPHA = M == 1 ? 1 : M + KW - 1;         // operand planes
    constexpr int TAPS = M == 1 ? KW : ALPHA;              // weight tiles per kernel row
    constexpr int CB = M == 1 ? 16 : 8;                    // channels per producer task
    constexpr int CHUNKS = kRowsChannels / CB;
    constexpr int HL = MODE == 1 ? 1 : 2;                  // halves of an operand
    constexpr int WIDE = MODE == 2 ? 2 : 1;                // accumulators per (tile, position)
    constexpr int kProducerWarps = kProducers<M>;
    constexpr int DEPTH = M == 1 ? 3 : 1;                  // tasks of a producer warp whose loads are in flight
    constexpr bool kRedo = M == 1 && MODE != 1;            // (one product keeps infinities; Winograd spreads them over its tiles in any case)
    static_assert(!SPLIT || MT == 1, "clusters share items of one tile");

    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t a_full[kRowsMaxA], a_empty[kRowsMaxA], b_full[kRowsMaxB], b_empty[kRowsMaxB];
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) float s_bias[kMaxSharedBias + 16];
    volatile int* abortp = &abort_flag;

    const int warp = ptx::uniform_warp(), lane = threadIdx.x & 31;
    const uint32_t a_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* const a_generic = smem_raw + (a_base - ptx::smem_u32(smem_raw));
    const uint32_t plane_bytes = (uint32_t)p.rows * 32u, a_slot_bytes = (uint32_t)(ALPHA * HL) * plane_bytes;
    const uint32_t b_tile_bytes = (uint32_t)p.bn * 32u, b_slot_bytes = (uint32_t)(TAPS * HL) * b_tile_bytes;
    const uint32_t b_base = a_base + (uint32_t)p.a_slots * a_slot_bytes;
    const int n_tasks = (p.rows_pad >> 5) * CHUNKS;        // producer tasks (32 cells x CB channels) per stage

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.a_slots; ++s) {
            ptx::mbar_init(ptx::smem_u32(&a_full[s]), (uint32_t)min(n_tasks, kProducerWarps));
            ptx::mbar_init(ptx::smem_u32(&a_empty[s]), 1);
        }
        for (int s = 0; s < p.b_slots; ++s) {
            ptx::mbar_init(ptx::smem_u32(&b_full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&b_empty[s]), 1);
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(ptx::smem_u32(&acc_full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&acc_empty[s]), kEpiWarps);
        }
        abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(ptx::smem_u32(&tmem_slot), (uint32_t)p.tmem_cols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = tmem_slot;
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();

    const uint32_t rank = SPLIT ? ptx::cluster_ctarank() : 0u;
    const unsigned first_item = SPLIT ? blockIdx.x / (unsigned)p.split : blockIdx.x;
    const unsigned item_step = SPLIT ? gridDim.x / (unsigned)p.split : gridDim.x;
    const int ks0 = SPLIT ? p.k_slots * (int)rank / p.split : 0, ks1 = SPLIT ? p.k_slots * ((int)rank + 1) / p.split : p.k_slots;
    const bool bias_in_smem = p.Cout <= kMaxSharedBias;
    if (bias_in_smem && warp >= kFirstEpi && warp < kFirstProducer) {
        for (int i = threadIdx.x - 32 * kFirstEpi; i < p.Cout; i += 32 * kEpiWarps) s_bias[i] = p.bias ? __ldg(p.bias + i) : 0.0f;
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");             // the epilogue warps only
    }

    if (warp == 0) {
        // ------------------------------ weight stream ------------------------------
        uint32_t bs = 0, b_phase = 0;
        bool ok = true;
        for (unsigned item = first_item; item < p.n_items && ok; item += item_step) {
            const unsigned nb = item / p.n_tile_blocks;
            const uint8_t* src = p.U + ((size_t)nb * p.k_slots + ks0) * p.steps * b_slot_bytes;
            const int steps = (ks1 - ks0) * p.steps;
            for (int s = 0; s < steps; ++s) {
                if (!ptx::mbar_wait_warp(ptx::smem_u32(&b_empty[bs]), b_phase ^ 1u, abortp)) {
                    ok = false;
                    break;
                }
                if (ptx::elect_one()) {
                    const uint32_t bar = ptx::smem_u32(&b_full[bs]);
                    ptx::mbar_expect_tx(bar, b_slot_bytes);
                    ptx::bulk_load(b_base + bs * b_slot_bytes, src + (size_t)s * b_slot_bytes, b_slot_bytes, bar);
                }
                if (++bs == (uint32_t)p.b_slots) {
                    bs = 0;
                    b_phase ^= 1u;
                }
            }
        }
        if (!ok && lane == 0) {
            if (!*abortp) atomicCAS(p.status, 0, kErrRowsStream);
            *abortp = 1;
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issue ------------------------------
        const uint32_t idesc = ptx::mma_idesc(1, 128, p.bn), idesc_wide = ptx::mma_idesc(1, 128, WIDE * p.bn);
        uint32_t as = 0, a_phase = 0, bs = 0, b_phase = 0, acc = 0, acc_phase = 0;
        int err = 0;
        const uint32_t a_lo0 = (1u << 16) | ((a_base & 0x3FFFFu) >> 4), b_lo0 = (1u << 16) | ((b_base & 0x3FFFFu) >> 4);
        const uint32_t plane16 = plane_bytes >> 4, tile16 = b_tile_bytes >> 4;
        for (unsigned item = first_item; item < p.n_items; item += item_step) {
            if (!ptx::mbar_wait_warp(ptx::smem_u32(&acc_empty[acc]), acc_phase ^ 1u, abortp)) {
                err = kErrRowsMmaAcc;
                goto failed;
            }
            ptx::tc_fence_after();
            const uint32_t d0 = tmem_base + acc * (uint32_t)(ALPHA * MT * WIDE * p.bn);
            uint32_t accumulate = 0;
            for (int ks = ks0; ks < ks1; ++ks) {
                if (!ptx::mbar_wait_warp(ptx::smem_u32(&a_full[as]), a_phase, abortp)) {
                    err = kErrRowsMmaA;
                    goto failed;
                }
                const uint32_t a_slot = a_lo0 + as * (a_slot_bytes >> 4);
                for (int v = 0; v < p.steps; ++v) {
                    const uint32_t a_lo = a_slot + (uint32_t)(v * p.step_rows) * 2u, b_lo = b_lo0 + bs * (b_slot_bytes >> 4);
                    if (!ptx::mbar_wait_warp(ptx::smem_u32(&b_full[bs]), b_phase, abortp)) {
                        err = kErrRowsMmaB;
                        goto failed;
                    }
                    ptx::tc_fence_after();
                    if (ptx::elect_one()) {
#pragma unroll
                        for (int pass = 0; pass < MODE; ++pass)
#pragma unroll
                            for (int t = 0; t < TAPS; ++t)
#pragma unroll
                                for (int mt = 0; mt < MT; ++mt) {
                                    const uint32_t a = a_lo + (M == 1 ? (uint32_t)(t * p.tap_rows) * 2u : (uint32_t)(t * HL) * plane16) + (pass == 1 ? plane16 : 0u) + (uint32_t)mt * 256u;
                                    const uint32_t b = b_lo + (uint32_t)(t * HL + (pass == 2 ? 1 : 0)) * tile16;
                                    const uint32_t d = d0 + (uint32_t)(((M == 1 ? 0 : t) * MT + mt) * WIDE) * (uint32_t)p.bn;
                                    ptx::mma_lo<1>(d, a, b, kDescHi, MODE == 2 && pass == 0 ? idesc_wide : idesc, (pass || (M == 1 && t)) ? 1u : accumulate);
                                }
                        ptx::mma_commit(ptx::smem_u32(&b_empty[bs]));
                    }
                    accumulate = 1u;
                    if (++bs == (uint32_t)p.b_slots) {
                        bs = 0;
                        b_phase ^= 1u;
                    }
                }
                if (ptx::elect_one()) ptx::mma_commit(ptx::smem_u32(&a_empty[as]));
                if (++as == (uint32_t)p.a_slots) {
                    as = 0;
                    a_phase ^= 1u;
                }
            }
            if (ptx::elect_one()) ptx::mma_commit(ptx::smem_u32(&acc_full[acc]));
            if (++acc == (uint32_t)p.acc_bufs) {
                acc = 0;
                acc_phase ^= 1u;
            }
        }
    failed:
        if (err && lane == 0) {
            if (!*abortp) atomicCAS(p.status, 0, err);
            *abortp = 1;
        }
    } else if (warp < kFirstProducer) {
        // ------------------------------ epilogue: A^T, bias, ReLU, store y ------------------------------
        const int q = warp & 3, part = (warp - kFirstEpi) >> 2;              // tensor-memory lane quarter; which half of the column chunks
        const long long ohw = (long long)p.OH * p.OW;
        const bool relu = p.relu != 0, pairs = M == 2 && (p.OW & 1) == 0 && (reinterpret_cast<uintptr_t>(p.y) & 7u) == 0;
        float2 check = make_float2(0.0f, 0.0f);
        uint32_t acc = 0, acc_phase = 0;
        for (unsigned item = first_item; item < p.n_items; item += item_step) {
            const unsigned nb = item / p.n_tile_blocks, tb = item - nb * p.n_tile_blocks;
            int got = 1;
            if (lane == 0) got = ptx::mbar_wait_relaxed(ptx::smem_u32(&acc_full[acc]), acc_phase, abortp) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) {
                if (lane == 0) {
                    if (!*abortp) atomicCAS(p.status, 0, kErrRowsEpilogue);
                    *abortp = 1;
                }
                break;
            }
            ptx::tc_fence_after();
            const int co0 = (int)nb * p.bn, n_co = min(p.bn, p.Cout - co0);
            for (int m = 0; m < MT; ++m) {
                const unsigned c = tb * (128u * MT) + (unsigned)m * 128u + (unsigned)(q * 32 + lane);
                const unsigned img = c / (unsigned)(p.Hq * p.Wq), r = c - img * (unsigned)(p.Hq * p.Wq);
                const int i = (int)(r / (unsigned)p.Wq), j = ((int)r - i * p.Wq) * M;
                const bool live = c < p.T && i < p.OH && j < p.OW;
                float* dst = p.y + (live ? ((size_t)img * p.Cout + co0) * ohw + (size_t)i * p.OW + j : 0);
                const bool second = M == 2 && j + 1 < p.OW;
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (acc * (uint32_t)(ALPHA * MT) + (uint32_t)m) * (uint32_t)(WIDE * p.bn);
                dst += (size_t)(part * 16) * ohw;
                for (int c0 = part * 16; c0 < n_co; c0 += 32) {
                    uint32_t v[ALPHA][16];
#pragma unroll
                    for (int xi = 0; xi < ALPHA; ++xi) ptx::tmem_ld16(taddr + (uint32_t)(xi * MT * WIDE * p.bn + c0), v[xi]);
                    if constexpr (WIDE == 2) {
                        uint32_t u[16];
#pragma unroll
                        for (int xi = 0; xi < ALPHA; ++xi) {
                            ptx::tmem_ld16(taddr + (uint32_t)((xi * MT * WIDE + 1) * p.bn + c0), u);
                            ptx::tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 16; ++e) v[xi][e] = __float_as_uint(__uint_as_float(v[xi][e]) + __uint_as_float(u[e]));
                        }
                    }
                    ptx::tmem_ld_wait();
                    float o[M][16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        if (M == 1) {
                            o[0][e] = __uint_as_float(v[0][e]);
                        } else {
#pragma unroll
                            for (int a = 0; a < M; ++a) {
                                float s = p.At[a * ALPHA] * __uint_as_float(v[0][e]);
#pragma unroll
                                for (int xi = 1; xi < ALPHA; ++xi) s = fmaf(p.At[a * ALPHA + xi], __uint_as_float(v[xi][e]), s);
                                o[a][e] = s;
                            }
                        }
                    }
                    if (SPLIT) {                                   // partial outputs over the operand slots, which nothing uses any more
                        float* red = reinterpret_cast<float*>(a_generic) + q * 32 + lane;
#pragma unroll
                        for (int e = 0; e < 16; ++e)
#pragma unroll
                            for (int a = 0; a < M; ++a) red[((c0 + e) * M + a) * 128] = o[a][e];
                        continue;
                    }
                    if (live) {
                        if constexpr (kRedo) {                         // no number from the first output on that is none
                            float2 t[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) t[e] = make_float2(o[0][2 * e], o[0][2 * e + 1]);
#pragma unroll
                            for (int d = 4; d > 0; d >>= 1)
#pragma unroll
                                for (int e = 0; e < d; ++e) t[e] = add_pair(t[e], t[e + d]);
                            check = add_pair(check, t[0]);
                        }
                        float bz[16];
                        if (bias_in_smem) {
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float4 b4 = *reinterpret_cast<const float4*>(s_bias + co0 + c0 + 4 * e);
                                bz[4 * e] = b4.x; bz[4 * e + 1] = b4.y; bz[4 * e + 2] = b4.z; bz[4 * e + 3] = b4.w;
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < 16; ++e) bz[e] = p.bias && c0 + e < n_co ? __ldg(p.bias + co0 + c0 + e) : 0.0f;
                        }
                        float* pj = dst;
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            if (c0 + e < n_co) {
                                float r0 = o[0][e] + bz[e], r1 = o[M - 1][e] + bz[e];
                                if (relu) {
                                    r0 = kRedo ? relu_nan(r0) : fmaxf(r0, 0.0f);
                                    r1 = kRedo ? relu_nan(r1) : fmaxf(r1, 0.0f);
                                }
                                if (pairs) {
                                    *reinterpret_cast<float2*>(pj) = make_float2(r0, r1);
                                } else {
                                    pj[0] = r0;
                                    if (second) pj[1] = r1;
                                }
                            }
                            pj += ohw;
                        }
                    }
                    dst += 32 * ohw;
                }
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&acc_empty[acc]));
            if (++acc == (uint32_t)p.acc_bufs) {
                acc = 0;
                acc_phase ^= 1u;
            }
        }
        if (kRedo && !SPLIT && !is_number(check.x + check.y)) {
            for (unsigned item = first_item; item < p.n_items; item += item_step) {
                const unsigned nb = item / p.n_tile_blocks, tb = item - nb * p.n_tile_blocks;
                for (int m = 0; m < MT; ++m) {
                    const unsigned c = tb * (128u * MT) + (unsigned)m * 128u + (unsigned)(q * 32 + lane);
                    const unsigned img = c / (unsigned)(p.Hq * p.Wq), r = c - img * (unsigned)(p.Hq * p.Wq);
                    const int i = (int)(r / (unsigned)p.Wq), j = (int)r - i * p.Wq;
                    if (c >= p.T || i >= p.OH || j >= p.OW) continue;
                    const int co0 = (int)nb * p.bn, n_co = min(p.bn, p.Cout - co0);
                    for (int c0 = part * 16; c0 < n_co; c0 += 32) rows_redo<TAPS>(p, img, i, j, nb, co0, c0, min(c0 + 16, n_co), 1);
                }
            }
        }
    } else {
        // ------------------------------ producers: x -> operand planes ------------------------------
        // A task is 32 cells (a lane each) x CB channels of one stage; the loads of a warp's next task are in flight while the
        // converted values of the current one wait for their slot.
        const int pw = warp - kFirstProducer;
        const size_t plane = (size_t)p.H * p.W;
        const int row_blocks = p.rows_pad >> 5;
        unsigned item = first_item;
        int ks = ks0, task = pw, decoded_block = -1;
        const float* base = p.x;
        unsigned inside = 0;                                         // positions of the cell's window inside the image
        auto decode = [&](int block) {
            const unsigned nb = item / p.n_tile_blocks, tb = item - nb * p.n_tile_blocks;
            const unsigned row = (unsigned)(block * 32 + lane), c = tb * (128u * MT) + row;
            const unsigned img = c / (unsigned)(p.Hq * p.Wq), r = c - img * (unsigned)(p.Hq * p.Wq);
            const int i = (int)(r / (unsigned)p.Wq), j = ((int)r - i * p.Wq) * M;
            const int ih = i - p.pad_h, iw = j - p.pad_w;
            inside = 0;
            if (row < (unsigned)p.rows && c < p.T && ih >= 0 && ih < p.H) {
#pragma unroll
                for (int e = 0; e < ALPHA; ++e)
                    if (iw + e >= 0 && iw + e < p.W) inside |= 1u << e;
            }
            base = inside ? p.x + (size_t)img * p.Cin * plane + (ptrdiff_t)ih * p.W + iw : p.x;
            decoded_block = block;
        };
        float d[DEPTH][CB][ALPHA];
        auto load = [&](float (&f)[CB][ALPHA]) {                     // the cursor's task; advances the cursor
            const int chunk = CHUNKS == 1 ? 0 : task / row_blocks, block = CHUNKS == 1 ? task : task - chunk * row_blocks;
            if (block != decoded_block) decode(block);
            const int c0 = ks * kRowsChannels + chunk * CB;
            const float* src = base + (size_t)c0 * plane;
            const int n_ch = p.Cin - c0;                             // channels of the task that exist (may exceed CB)
#pragma unroll
            for (int ch = 0; ch < CB; ++ch) {
#pragma unroll
                for (int e = 0; e < ALPHA; ++e) f[ch][e] = ch < n_ch && ((inside >> e) & 1u) ? __ldg(src + e) : 0.0f;
                src += plane;
            }
            task += kProducerWarps;
            if (task >= n_tasks) {
                task = pw;
                if (++ks == ks1) {
                    ks = ks0;
                    item += item_step;
                    decoded_block = -1;
                }
            }
        };
        const int per_stage = pw < n_tasks ? (n_tasks - pw + kProducerWarps - 1) / kProducerWarps : 0;
        const long long n_local = first_item < p.n_items ? (p.n_items - first_item + item_step - 1) / item_step : 0;
        const long long total = n_local * (ks1 - ks0) * per_stage;
        uint32_t as = 0, a_phase = 0;
        int in_stage = 0;                                            // tasks of the current stage already stored
        bool ok = true;
#pragma unroll
        for (int b = 0; b < DEPTH; ++b)
            if (b < total) load(d[b]);
        for (long long it = 0; it < total && ok; it += DEPTH) {
#pragma unroll
            for (int b = 0; b < DEPTH; ++b) {
                if (it + b >= total) break;
                if (in_stage == 0) {
                    int got = 1;
                    if (lane == 0) got = ptx::mbar_wait_relaxed(ptx::smem_u32(&a_empty[as]), a_phase ^ 1u, abortp) ? 1 : 0;
                    got = __shfl_sync(0xffffffffu, got, 0);
                    if (!got) {
                        if (lane == 0) {
                            if (!*abortp) atomicCAS(p.status, 0, kErrRowsProducer);
                            *abortp = 1;
                        }
                        ok = false;
                        break;
                    }
                }
                const int my_task = pw + in_stage * kProducerWarps;
                const int chunk = CHUNKS == 1 ? 0 : my_task / row_blocks, row = (my_task - chunk * row_blocks) * 32 + lane;
                uint8_t* const dst = a_generic + as * a_slot_bytes + row * 32;
                const int flip = (row >> 2) & 1;
                const bool in_plane = row < p.rows;
#pragma unroll
                for (int g = 0; g < CB / 8; ++g) {
                    float v[8][ALPHA];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const float* f = d[b][8 * g + u];
                        if constexpr (M == 1) {
                            v[u][0] = f[0];
                        } else {                                     // alpha = 4: rows (a 0 b 0), (0 a b 0), (0 a b 0), (0 a 0 b) of B^T
                            v[u][0] = fmaf(p.Bt[0], f[0], p.Bt[2] * f[2]);
                            v[u][1] = fmaf(p.Bt[5], f[1], p.Bt[6] * f[2]);
                            v[u][2] = fmaf(p.Bt[9], f[1], p.Bt[10] * f[2]);
                            v[u][3] = fmaf(p.Bt[13], f[1], p.Bt[15] * f[3]);
                        }
                    }
                    const int piece = ((chunk + g) ^ flip) << 4;
#pragma unroll
                    for (int xi = 0; xi < ALPHA; ++xi) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            const float a = v[2 * h][xi], c = v[2 * h + 1][xi];
                            hi[h] = pack_bf16(a, c);
                            lo[h] = HL == 2 ? pack_bf16(a - __uint_as_float(hi[h] << 16), c - __uint_as_float(hi[h] & 0xffff0000u)) : 0u;
                        }
                        if (in_plane) {
                            *reinterpret_cast<uint4*>(dst + (HL * xi) * plane_bytes + piece) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                            if (HL == 2) *reinterpret_cast<uint4*>(dst + (HL * xi + 1) * plane_bytes + piece) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                        }
                    }
                }
                if (++in_stage == per_stage) {
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // the tensor core reads these through the async proxy
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&a_full[as]));
                    in_stage = 0;
                    if (++as == (uint32_t)p.a_slots) {
                        as = 0;
                        a_phase ^= 1u;
                    }
                }
                // (behind the fence, which waits for the loads in flight)
                if (it + b + DEPTH < total) load(d[b]);
            }
        }
    }

    if (SPLIT) {
        __syncwarp();
        ptx::cluster_sync_all();
        if (warp >= kFirstEpi && warp < kFirstEpi + 16 && !*abortp && first_item < p.n_items) {           // four sets of four warps share the columns
            const unsigned nb = first_item / p.n_tile_blocks, tb = first_item - nb * p.n_tile_blocks;
            const int rw = (warp & 3) * 32 + lane, co0 = (int)nb * p.bn;
            const unsigned c = tb * 128u + (unsigned)rw;
            const unsigned img = c / (unsigned)(p.Hq * p.Wq), r = c - img * (unsigned)(p.Hq * p.Wq);
            const int i = (int)(r / (unsigned)p.Wq), j = ((int)r - i * p.Wq) * M;
            if (c < p.T && i < p.OH && j < p.OW) {
                const long long ohw = (long long)p.OH * p.OW;
                float* const dst = p.y + ((size_t)img * p.Cout + co0) * ohw + (size_t)i * p.OW + j;
                float check = 0.0f;
                ptx::cluster_reduce_columns(a_base, p.bn * M, rank, p.split, rw, (warp - kFirstEpi) >> 2, 4, [&](int col, float sum) {
                    const int co = col / M, a = col - co * M;
                    if (co0 + co >= p.Cout || (M == 2 && j + a >= p.OW)) return;
                    sum += p.bias ? __ldg(p.bias + co0 + co) : 0.0f;
                    if (kRedo) check += sum;
                    dst[(long long)co * ohw + a] = !p.relu ? sum : kRedo ? relu_nan(sum) : fmaxf(sum, 0.0f);
                });
                if (kRedo && !is_number(check))
                    rows_redo<TAPS>(p, img, i, j, nb, co0, p.bn * (int)rank / p.split + ((warp - kFirstEpi) >> 2), min(p.bn * ((int)rank + 1) / p.split, p.Cout - co0), 4);
            }
        }
        __syncwarp();
        ptx::cluster_sync_all();                           // nobody leaves while its partial sums are being read
    }

    // Teardown.  After an aborted run give copies still in flight time to land before shared memory is released.
    if (*abortp) __nanosleep(200000);
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

struct WeightParams {
    const float* w;
    uint8_t* U;
    int Cout, Cin, steps, per_step, k_slots, bn, n_co_blocks, m, alpha, taps, halves;
    float G[kRowsMaxAlpha * 7];
};

// A thread per (output channel row of a tile, input channel), all weight tiles of one kernel row: U [channel block][stage][kernel
// row][tile][hi, lo][bn rows of 32 bytes, swizzled].
__global__ void __launch_bounds__(256) rows_weights_kernel(const __grid_constant__ WeightParams p)
{
    const long long gid = (long long)blockIdx.x * 256 + threadIdx.x;
    const long long total = (long long)p.n_co_blocks * p.k_slots * p.steps * p.bn * kRowsChannels;
    if (gid >= total) return;
    const int c = (int)(gid % kRowsChannels);
    long long r = gid / kRowsChannels;
    const int row = (int)(r % p.bn);
    r /= p.bn;
    const int v = (int)(r % p.steps);
    r /= p.steps;
    const int ks = (int)(r % p.k_slots), nb = (int)(r / p.k_slots);
    const int co = nb * p.bn + row, ci = ks * kRowsChannels + c;
    const bool ok = co < p.Cout && ci < p.Cin;
    const float* src = p.w + (((size_t)(ok ? co : 0) * p.Cin + (ok ? ci : 0)) * p.steps + v) * p.per_step;
    const size_t tile = (size_t)p.bn * 32;
    uint8_t* dst = p.U + (((size_t)nb * p.k_slots + ks) * p.steps + v) * p.taps * p.halves * tile + row * 32 + (((c >> 3) ^ ((row >> 2) & 1)) << 4) + (c & 7) * 2;
    for (int t = 0; t < p.taps; ++t) {
        float s = 0.0f;
        if (ok) {
            if (p.m == 1) {
                s = src[t];
            } else {
                for (int b = 0; b < p.per_step; ++b) s = fmaf(p.G[t * p.per_step + b], src[b], s);
            }
        }
        __nv_bfloat16 h = __float2bfloat16_rn(s);
        float lo = s - __bfloat162float(h);
        if (p.halves == 2 && !is_number(lo)) {                     // hi is infinite: a finite weight is cut instead of rounded up, an infinite one is all hi
            if (is_number(s)) h = __float2bfloat16_rz(s);
            lo = is_number(s) ? s - __bfloat162float(h) : 0.0f;
        }
        *reinterpret_cast<__nv_bfloat16*>(dst + (p.halves * t) * tile) = h;
        if (p.halves == 2) *reinterpret_cast<__nv_bfloat16*>(dst + (2 * t + 1) * tile) = __float2bfloat16_rn(lo);
    }
}

typedef void (*RowsKernel)(RowsParams);

template <int KW, int MODE>
RowsKernel rows_kernel_mode(const RowsPlan& p)
{
    if (p.mt == 2) return rows_conv_kernel<1, KW, 2, MODE, false>;
    if constexpr (MODE != 3 || KW < 5)
        if (p.split > 1) return rows_conv_kernel<1, KW, 1, MODE, true>;
    if constexpr (MODE != 3 || KW < 7)
        if (p.split == 1) return rows_conv_kernel<1, KW, 1, MODE, false>;
    return nullptr;                                          // (no plan has it)
}

template <int KW>
RowsKernel rows_kernel_of(const RowsPlan& p)
{
    return p.mode == 1 ? rows_kernel_mode<KW, 1>(p) : p.mode == 2 ? rows_kernel_mode<KW, 2>(p) : rows_kernel_mode<KW, 3>(p);
}

RowsKernel rows_kernel(const RowsPlan& p)
{
    if (p.s.m == 2) return p.split > 1 ? rows_conv_kernel<2, 3, 1, 3, true> : rows_conv_kernel<2, 3, 1, 3, false>;
    switch (p.taps) {
        case 2: return rows_kernel_of<2>(p);
        case 3: return rows_kernel_of<3>(p);
        case 5: return rows_kernel_of<5>(p);
        case 7: return rows_kernel_of<7>(p);
        default: return nullptr;
    }
}

}  // namespace

bool rows_matrices_ok(const RowsConv& rc)
{
    if (rc.p.s.m == 1) return true;
    const float* b = rc.Bt;
    return b[1] == 0.0f && b[3] == 0.0f && b[4] == 0.0f && b[7] == 0.0f && b[8] == 0.0f && b[11] == 0.0f && b[12] == 0.0f && b[14] == 0.0f;
}

cudaError_t rows_setup(RowsConv* rc)
{
    rc->ready = false;
    const RowsKernel kern = rows_kernel(rc->p);
    if (!kern) return cudaErrorInvalidValue;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&rc->num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsSmemBytes);
    rc->ready = e == cudaSuccess;
    return e;
}

cudaError_t launch_rows_weights(const RowsConv& rc, const float* w, void* U, cudaStream_t stream)
{
    WeightParams p = {};
    const RowsPlan& rp = rc.p;
    p.w = w;
    p.U = static_cast<uint8_t*>(U);
    p.Cout = rp.s.Cout; p.Cin = rp.s.Cin; p.steps = rp.steps; p.per_step = rp.s.kh * rp.s.kw / rp.steps; p.k_slots = rp.k_slots; p.bn = rp.bn; p.n_co_blocks = rp.n_co_blocks;
    p.m = rp.s.m; p.alpha = rp.alpha; p.taps = rp.taps; p.halves = rp.mode == 1 ? 1 : 2;
    for (int i = 0; i < rp.alpha * rp.s.kw && rp.s.m > 1; ++i) p.G[i] = rc.G[i];
    const long long total = (long long)p.n_co_blocks * p.k_slots * p.steps * p.bn * kRowsChannels;
    rows_weights_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_rows_conv(const RowsConv& rc, const float* x, const void* U, const float* bias, float* y, int relu, int* status,
                             cudaStream_t stream)
{
    if (!rc.ready) return cudaErrorInvalidValue;
    const RowsPlan& rp = rc.p;
    RowsParams p = {};
    p.x = x; p.bias = bias; p.y = y; p.U = static_cast<const uint8_t*>(U); p.status = status;
    p.T = (unsigned)rp.T; p.n_items = (unsigned)rp.n_items; p.n_tile_blocks = (unsigned)rp.n_tile_blocks;
    p.Cin = rp.s.Cin; p.Cout = rp.s.Cout; p.H = rp.s.H; p.W = rp.s.W; p.OH = rp.s.OH; p.OW = rp.s.OW; p.steps = rp.steps; p.step_rows = rp.step_rows; p.tap_rows = rp.tap_rows; p.taps_down = rp.s.kw == 1 ? 1 : 0; p.pad_h = rp.s.pad_h; p.pad_w = rp.s.pad_w;
    p.Hq = rp.Hq; p.Wq = rp.Wq; p.rows = rp.rows; p.rows_pad = rp.rows_pad; p.k_slots = rp.k_slots; p.bn = rp.bn;
    p.a_slots = rp.a_slots; p.b_slots = rp.b_slots; p.acc_bufs = rp.acc_bufs; p.split = rp.split; p.relu = relu;
    p.tmem_cols = 32;
    while (p.tmem_cols < rp.acc_bufs * rp.n_acc * rp.mt * (rp.mode == 2 ? 2 : 1) * rp.bn) p.tmem_cols *= 2;
    if (rp.s.m > 1) {
        for (int i = 0; i < rp.alpha * rp.alpha; ++i) p.Bt[i] = rc.Bt[i];
        for (int i = 0; i < rp.s.m * rp.alpha; ++i) p.At[i] = rc.At[i];
    }
    const RowsKernel kern = rows_kernel(rp);
    const dim3 block(rp.s.m == 1 ? kRowsThreads<1> : kRowsThreads<2>);
    // (the full budget: at most one CTA per SM, so that tensor memory is never contended)
    if (rp.split > 1) return launch_cluster(rp.split, kern, dim3((unsigned)(rp.n_items * rp.split)), block, (size_t)kRowsSmemBytes, stream, p);
    const unsigned grid = rp.n_items < rc.num_sms ? (unsigned)rp.n_items : (unsigned)rc.num_sms;
    return launch_overlapped(kern, dim3(grid), block, (size_t)kRowsSmemBytes, stream, p);
}

}  // namespace mnnb
