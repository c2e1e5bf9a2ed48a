// Packed-line convolution: the GEMM scheme for strided, dilated and few-channel layers as a tensor-core product whose left
// operand is staged once per region and read at shifted start rows (line_plan.h).
//
//     y[co][cell] = sum over (element block, tap) of  A[plane][cell + shift(tap)][element] * U[tap][co][element]
//
// Two launches.  The pack kernel transposes x into planes of positions, rounded to TF32 or BF16.  The product kernel is the
// persistent pipeline of contract_umma.cu (TMA producer, one MMA thread, epilogue warps, two accumulators) with two rings: a
// region of 128 * mt + span consecutive positions x 32 elements is staged once per (element block, plane), and one weight
// tile per tap.  A row of the region is 128 bytes in the 128-byte swizzle, whose pattern depends on the address alone and
// whose 8-row groups lie 1024 bytes apart, so row r of the operand is r * 128 bytes behind any start row: a tap is a start
// address, and an input element crosses from L2 once per region instead of k * k times.
//
// What bounds it: the tensor core's TF32 rate and the issuing warp (3 x 3 dilation 2, 256 channels 28 x 28, batch 16:
// 29 us product, 510 TFLOP/s); on few-channel layers the bytes of the packed planes.  Measured, both
// launches, against the implicit gather / the patch matrix: that layer 37 us (86 / 107); 64 -> 128 3x3 stride 2 at 56 x 56
// batch 32 27 us (45 / 66); 128 -> 256 at 28 x 28 26 us (45 / 56); 256 -> 512 at 14 x 14 38 us (79 / 68); 3 -> 64 7x7
// stride 2 at 224 x 224 batch 32 70 us (247 / 156).
//
// BF16 operands (the BF16 accuracy class) halve the planes and the instructions: 256 channels 56 x 56 batch 64 product 303 ->
// 176 us (1.35 PFLOP/s), layer 248 us against 431 in the Winograd scheme in a warm loop, 303 against 451 with cold inputs; 64
// channels 56 x 56 batch 64 50 us against 103 (warm).  Error against 64 bits 2.35e-3, Winograd F(4 x 4) on TF32 3.20e-3.
#include "line_conv.h"

#include <cuda_bf16.h>

#include <type_traits>

#include "contract_umma.h"
#include "umma.cuh"

namespace mnnb {

namespace {

constexpr int kEpiWarps = 8;
constexpr int kMaxSharedBias = 2048;     // output channels whose bias is staged (+ 16 of slack for reads past the last)
constexpr int line_threads(int mt) { return 32 * (1 + mt + kEpiWarps); }      // producer, one issuing warp per tile, epilogue
constexpr int kErrLineProducer = 51, kErrLineMmaA = 52, kErrLineMmaB = 53, kErrLineMmaAcc = 54, kErrLineEpilogue = 55;

struct LineParams {
    const float* bias;
    float* y;
    int* status;
    long long T;
    unsigned n_items, n_tile_blocks;
    int Cout, bn, blocks, n_groups, region, boxes, box_rows, a_slots, b_slots, tmem_cols;
    int strips, Hq, Wq, OH, OW, relu;
    int group_plane[kLineMaxPlanes], group_base[kLineMaxPlanes], group_first[kLineMaxPlanes], group_taps[kLineMaxPlanes];
    int tap_rel[kLineMaxTaps];
};

// Shared-memory descriptors of 128-byte rows in the 128-byte swizzle (ptx::smem_desc_k128) as low words over a common high
// word, so that an instruction costs the issuing thread one addition per operand.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);

// MT = tiles of 128 cells per item, KS = tensor-core steps per block of elements, G = weight tiles per step (slot, barrier and
// commit), all fixed at compile time, with one issuing warp per tile of cells.  The issuing warp is on the critical path:
// dilation-2 layer above, product only: 66 us with run-time loop bounds, 43.5 unrolled, 38 with up to three taps per step;
// 256 -> 512 stride 2: 36 -> 31 us with the failure checks out of the loop conditions; then 38.1 -> 26.8 us for both kernels
// with the loops run by the whole warp and one elected lane issuing (dilation-2 layer 38.3 -> 36.1, both kernels).
template <int MT, int KS, int G, bool BF16>
__global__ void __launch_bounds__(line_threads(MT), 1)
line_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_u, const __grid_constant__ LineParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t a_full[kLineMaxA], a_empty[kLineMaxA], b_full[kLineMaxB], b_empty[kLineMaxB];
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) float s_bias[kMaxSharedBias + 16];
    volatile int* abortp = &abort_flag;

    const int warp = ptx::uniform_warp(), lane = threadIdx.x & 31;
    constexpr int kBlockElems = BF16 ? 64 : 32;
    const uint32_t a_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_slot_bytes = (uint32_t)p.region * 128u, b_tile_bytes = (uint32_t)p.bn * 128u, b_slot_bytes = G * b_tile_bytes;
    const uint32_t b_base = a_base + (uint32_t)p.a_slots * a_slot_bytes;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.a_slots; ++s) {
            ptx::mbar_init(ptx::smem_u32(&a_full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&a_empty[s]), MT);
        }
        for (int s = 0; s < p.b_slots; ++s) {
            ptx::mbar_init(ptx::smem_u32(&b_full[s]), 1);
            ptx::mbar_init(ptx::smem_u32(&b_empty[s]), MT);
        }
        for (int s = 0; s < 2; ++s) {
            ptx::mbar_init(ptx::smem_u32(&acc_full[s]), MT);
            ptx::mbar_init(ptx::smem_u32(&acc_empty[s]), kEpiWarps);
        }
        abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::prefetch_tensormap(&map_a);
        ptx::prefetch_tensormap(&map_u);
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
    const bool bias_in_smem = p.Cout <= kMaxSharedBias;
    if (bias_in_smem && warp > MT) {
        for (int i = threadIdx.x - 32 * (1 + MT); i < p.Cout; i += 32 * kEpiWarps) s_bias[i] = p.bias ? __ldg(p.bias + i) : 0.0f;
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");            // the epilogue warps only
    }

    if (warp == 0) {
        // ------------------------------ regions of A and weight tiles ------------------------------
        {
            uint32_t as = 0, a_phase = 0, bs = 0, b_phase = 0;
            bool ok = true;
            for (unsigned item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
                const unsigned nb = item / p.n_tile_blocks, tb = item - nb * p.n_tile_blocks;
                for (int eb = 0; eb < p.blocks && ok; ++eb)
                    for (int g = 0; g < p.n_groups && ok; ++g) {
                        if (!ptx::mbar_wait_warp(ptx::smem_u32(&a_empty[as]), a_phase ^ 1u, abortp)) {
                            ok = false;
                            break;
                        }
                        const uint32_t abar = ptx::smem_u32(&a_full[as]);
                        const int row0 = (int)(tb * 128u * (unsigned)MT) + p.group_base[g];
                        if (ptx::elect_one()) {
                            ptx::mbar_expect_tx(abar, a_slot_bytes);
                            for (int b = 0; b < p.boxes; ++b)
                                ptx::tma_load_3d(a_base + as * a_slot_bytes + (uint32_t)(b * p.box_rows) * 128u, &map_a, abar, eb * kBlockElems,
                                                 row0 + b * p.box_rows, p.group_plane[g]);
                        }
                        if (++as == (uint32_t)p.a_slots) {
                            as = 0;
                            a_phase ^= 1u;
                        }
                        const int t0 = p.group_first[g], t1 = t0 + p.group_taps[g];
                        for (int t = t0; t < t1; t += G) {
                            if (!ptx::mbar_wait_warp(ptx::smem_u32(&b_empty[bs]), b_phase ^ 1u, abortp)) {
                                ok = false;
                                break;
                            }
                            const uint32_t bbar = ptx::smem_u32(&b_full[bs]);
                            const int n = min(G, t1 - t);
                            if (ptx::elect_one()) {
                                ptx::mbar_expect_tx(bbar, (uint32_t)n * b_tile_bytes);
#pragma unroll
                                for (int j = 0; j < G; ++j)
                                    if (j < n)
                                        ptx::tma_load_3d(b_base + bs * b_slot_bytes + j * b_tile_bytes, &map_u, bbar, eb * kBlockElems, (int)nb * p.bn, t + j);
                            }
                            if (++bs == (uint32_t)p.b_slots) {
                                bs = 0;
                                b_phase ^= 1u;
                            }
                        }
                    }
            }
            if (!ok && lane == 0) {
                if (!*abortp) atomicCAS(p.status, 0, kErrLineProducer);
                *abortp = 1;
            }
        }
    } else if (warp <= MT) {
        // ------------------------------ MMA issue: one warp per tile of 128 cells ------------------------------
        {
            const uint32_t tile = (uint32_t)warp - 1u;
            const uint32_t idesc = ptx::mma_idesc(BF16 ? 1 : 2, 128, p.bn);
            uint32_t as = 0, a_phase = 0, bs = 0, b_phase = 0, acc = 0, acc_phase = 0;
            int err = 0;
            const uint32_t a_lo_base = (1u << 16) | (((a_base & 0x3FFFFu) >> 4) + tile * 1024u), b_lo_base = (1u << 16) | ((b_base & 0x3FFFFu) >> 4);
            for (unsigned item = blockIdx.x; item < p.n_items; item += gridDim.x) {
                if (!ptx::mbar_wait_warp(ptx::smem_u32(&acc_empty[acc]), acc_phase ^ 1u, abortp)) {
                    err = kErrLineMmaAcc;
                    goto failed;
                }
                ptx::tc_fence_after();
                const uint32_t d0 = tmem_base + (acc * MT + tile) * (uint32_t)p.bn;
                uint32_t accumulate = 0;
                for (int eb = 0; eb < p.blocks; ++eb)
                    for (int g = 0; g < p.n_groups; ++g) {
                        const int t0 = p.group_first[g], t1 = t0 + p.group_taps[g];
                        const uint32_t a_lo_slot = a_lo_base + as * (a_slot_bytes >> 4);
                        if (!ptx::mbar_wait_warp(ptx::smem_u32(&a_full[as]), a_phase, abortp)) {
                            err = kErrLineMmaA;
                            goto failed;
                        }
                        for (int t = t0; t < t1; t += G) {
                            const int n = min(G, t1 - t);
                            uint32_t a_lo[G];
#pragma unroll
                            for (int j = 0; j < G; ++j) a_lo[j] = a_lo_slot + (uint32_t)p.tap_rel[j < n ? t + j : t] * 8u;
                            const uint32_t b_lo = b_lo_base + bs * (b_slot_bytes >> 4);
                            if (!ptx::mbar_wait_warp(ptx::smem_u32(&b_full[bs]), b_phase, abortp)) {
                                err = kErrLineMmaB;
                                goto failed;
                            }
                            if (ptx::elect_one()) {
#pragma unroll
                                for (int j = 0; j < G; ++j)
                                    if (j < n) {
#pragma unroll
                                        for (int ks = 0; ks < KS; ++ks)
                                            ptx::mma_lo<BF16 ? 1 : 0>(d0, a_lo[j] + (uint32_t)(ks * 2), b_lo + (uint32_t)j * (b_tile_bytes >> 4) + (uint32_t)(ks * 2), kDescHi,
                                                                      idesc, (j | ks) ? 1u : accumulate);
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
                acc ^= 1u;
                if (acc == 0) acc_phase ^= 1u;
            }
        failed:
            if (err && lane == 0) {
                if (!*abortp) atomicCAS(p.status, 0, err);
                *abortp = 1;
            }
        }
    } else {
        // ------------------------------ epilogue: bias, ReLU, store y ------------------------------
        const int q = warp & 3, part = (warp - 1 - MT) >> 2;                 // tensor-memory lane quarter; which half of the column chunks
        const long long ohw = (long long)p.OH * p.OW;
        const bool relu = p.relu != 0;
        uint32_t acc = 0, acc_phase = 0;
        for (unsigned item = blockIdx.x; item < p.n_items; item += gridDim.x) {
            const unsigned nb = item / p.n_tile_blocks, tb = item - nb * p.n_tile_blocks;
            int got = 1;
            if (lane == 0) got = ptx::mbar_wait_relaxed(ptx::smem_u32(&acc_full[acc]), acc_phase, abortp) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) {
                if (lane == 0) {
                    if (!*abortp) atomicCAS(p.status, 0, kErrLineEpilogue);
                    *abortp = 1;
                }
                break;
            }
            ptx::tc_fence_after();
            const int co0 = (int)nb * p.bn, n_co = min(p.bn, p.Cout - co0), n_chunks = (n_co + 15) >> 4;
            for (int m = 0; m < MT; ++m) {
                const long long cell = (long long)tb * (128 * MT) + m * 128 + q * 32 + lane;
                bool live = cell < p.T;
                const unsigned c = live ? (unsigned)cell : 0u;          // (T < 2^31)
                const unsigned n = c / (unsigned)(p.Hq * p.Wq), r = c - n * (unsigned)(p.Hq * p.Wq);
                const unsigned img = n / (unsigned)p.strips;
                const unsigned i = r / (unsigned)p.Wq, j = r - i * (unsigned)p.Wq + (n - img * (unsigned)p.strips) * (unsigned)p.Wq;
                live = live && (int)i < p.OH && (int)j < p.OW;
                float* const dst = p.y + ((size_t)img * p.Cout + co0) * ohw + (live ? (size_t)i * p.OW + j : 0);
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + acc * (uint32_t)(MT * p.bn) + (uint32_t)(m * p.bn);
                auto store = [&](const uint32_t (&v)[16], int ch) {
                    if (!live) return;
                    float* pj = dst + (size_t)(ch * 16) * ohw;
                    const int left = n_co - ch * 16;
                    float bz[16];
                    if (bias_in_smem) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float4 b4 = *reinterpret_cast<const float4*>(s_bias + co0 + ch * 16 + 4 * e);
                            bz[4 * e] = b4.x; bz[4 * e + 1] = b4.y; bz[4 * e + 2] = b4.z; bz[4 * e + 3] = b4.w;
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e) bz[e] = (p.bias && e < left) ? __ldg(p.bias + co0 + ch * 16 + e) : 0.0f;
                    }
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        if (e < left) {
                            const float o = __uint_as_float(v[e]) + bz[e];
                            *pj = relu ? fmaxf(o, 0.0f) : o;
                        }
                        pj += ohw;
                    }
                };
                uint32_t va[16], vb[16];
                if (part < n_chunks) ptx::tmem_ld16(taddr + (uint32_t)(part * 16), va);
                for (int ch = part; ch < n_chunks; ch += 4) {
                    ptx::tmem_ld_wait();
                    if (ch + 2 < n_chunks) ptx::tmem_ld16(taddr + (uint32_t)((ch + 2) * 16), vb);
                    store(va, ch);
                    if (ch + 2 < n_chunks) {
                        ptx::tmem_ld_wait();
                        if (ch + 4 < n_chunks) ptx::tmem_ld16(taddr + (uint32_t)((ch + 4) * 16), va);
                        store(vb, ch + 2);
                    }
                }
            }
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&acc_empty[acc]));
            acc ^= 1u;
            if (acc == 0) acc_phase ^= 1u;
        }
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

// ---------------------------------------------------------------------------
// Packing x.
// ---------------------------------------------------------------------------
struct PackParams {
    const float* x;
    void* A;
    long long P, T;
    int Cin, H, W, k, stride, dil, pad, strips, Hq, Wq, elems, n_planes;
    int phase_h[kLineMaxPlanes], phase_w[kLineMaxPlanes];
};

__device__ __forceinline__ float tf32_rn(float v)
{
    uint32_t u;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(v));
    return __uint_as_float(u);
}

// 32 positions x 64 channels of one plane per CTA, transposed through shared memory: lanes run over positions while x is
// read and over channels while A is written.  The planes of a position block are neighbours in the grid, so that the phases
// of a stride share the sectors of x in L2.
template <bool BF16>
__global__ void __launch_bounds__(256) line_pack_kernel(const __grid_constant__ PackParams p)
{
    __shared__ float tile[64][33];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int z = blockIdx.x % p.n_planes;
    const long long p0 = (long long)(blockIdx.x / p.n_planes) * 32;
    const int c0 = blockIdx.y * 64;
    {
        const long long pos = p0 + lane;
        const unsigned c = pos < p.T ? (unsigned)pos : 0u;
        const unsigned n = c / (unsigned)(p.Hq * p.Wq), r = c - n * (unsigned)(p.Hq * p.Wq);
        const unsigned i = r / (unsigned)p.Wq, j = r - i * (unsigned)p.Wq;
        const int ih = (int)i * p.stride + p.phase_h[z] - p.pad, iw = (int)j * p.stride + p.phase_w[z] - p.pad;
        const bool ok = pos < p.T && ih >= 0 && ih < p.H && iw >= 0 && iw < p.W;
        const size_t plane = (size_t)p.H * p.W;
        const float* src = p.x + ((size_t)n * p.Cin + c0 + warp) * plane + (ok ? (size_t)ih * p.W + iw : 0);
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = ok && c0 + warp + 8 * e < p.Cin ? __ldg(src + (size_t)(8 * e) * plane) : 0.0f;
#pragma unroll
        for (int e = 0; e < 8; ++e) tile[warp + 8 * e][lane] = BF16 ? v[e] : tf32_rn(v[e]);
    }
    __syncthreads();
    // 16 lanes write the 64 channels of a position, four each
    const int cv = (threadIdx.x & 15) * 4;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int pl = (threadIdx.x >> 4) + 16 * h;
        const long long pos = p0 + pl;
        if (pos >= p.P || c0 + cv >= p.elems) continue;
        const long long at = ((long long)z * p.P + pos) * p.elems + c0 + cv;
        if (BF16) {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(tile[cv][pl], tile[cv + 1][pl]), hi = __floats2bfloat162_rn(tile[cv + 2][pl], tile[cv + 3][pl]);
            *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.A) + at) =
                make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        } else {
            *reinterpret_cast<float4*>(static_cast<float*>(p.A) + at) = make_float4(tile[cv][pl], tile[cv + 1][pl], tile[cv + 2][pl], tile[cv + 3][pl]);
        }
    }
}

// Few channels: a warp gathers the elements (ci, b) of 32 positions, a position per lane, and writes them as rows of 128 bytes
// through shared memory (only the elements the tensor core reads; the rest of a row is never read).
template <int USED>
__global__ void __launch_bounds__(256) line_pack_few_kernel(const __grid_constant__ PackParams p)
{
    __shared__ __align__(16) float tile[8][32][USED + 4];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int z = blockIdx.y;
    const long long p0 = (long long)blockIdx.x * 256 + warp * 32;
    const long long pos = p0 + lane;
    const unsigned c = pos < p.T ? (unsigned)pos : 0u;
    const unsigned n = c / (unsigned)(p.Hq * p.Wq), r = c - n * (unsigned)(p.Hq * p.Wq);
    const unsigned img = n / (unsigned)p.strips;
    const unsigned i = r / (unsigned)p.Wq, j = r - i * (unsigned)p.Wq + (n - img * (unsigned)p.strips) * (unsigned)p.Wq;
    const int ih = (int)i * p.stride + p.phase_h[z] - p.pad, iw0 = (int)j * p.stride - p.pad;
    const bool row_ok = pos < p.T && ih >= 0 && ih < p.H;
    const size_t plane = (size_t)p.H * p.W;
    const float* src = p.x + (size_t)img * p.Cin * plane + (row_ok ? (size_t)ih * p.W : 0);
    unsigned cols = 0;                                                  // kernel columns inside the image
    for (int b = 0; b < p.k; ++b)
        if (row_ok && iw0 + b * p.dil >= 0 && iw0 + b * p.dil < p.W) cols |= 1u << b;
    int ci = 0, b = 0;
    float v[USED];
#pragma unroll
    for (int e = 0; e < USED; ++e) {
        v[e] = ci < p.Cin && ((cols >> b) & 1u) ? __ldg(src + (size_t)ci * plane + iw0 + b * p.dil) : 0.0f;
        if (++b == p.k) {
            b = 0;
            ++ci;
        }
    }
#pragma unroll
    for (int q = 0; q < USED / 4; ++q)
        *reinterpret_cast<float4*>(&tile[warp][lane][4 * q]) =
            make_float4(tf32_rn(v[4 * q]), tf32_rn(v[4 * q + 1]), tf32_rn(v[4 * q + 2]), tf32_rn(v[4 * q + 3]));
    __syncwarp();
    float* dst = static_cast<float*>(p.A) + ((long long)z * p.P + p0) * 32;
    const int piece = lane & 7;
    if (piece < USED / 4)
#pragma unroll
        for (int q = 0; q < 32; q += 4) {
            const int row = q + (lane >> 3);
            if (p0 + row < p.P) *reinterpret_cast<float4*>(dst + row * 32 + piece * 4) = *reinterpret_cast<const float4*>(&tile[warp][row][piece * 4]);
        }
}

struct WeightParams {
    const float* w;
    void* U;
    int Cout, Cin, k, elems, few, bf16, n_taps;
    int tap_id[kLineMaxTaps];
};

__global__ void __launch_bounds__(256) line_weights_kernel(const __grid_constant__ WeightParams p)
{
    const long long gid = (long long)blockIdx.x * 256 + threadIdx.x;
    if (gid >= (long long)p.n_taps * p.Cout * p.elems) return;
    const int e = (int)(gid % p.elems);
    const long long r = gid / p.elems;
    const int co = (int)(r % p.Cout), tap = p.tap_id[r / p.Cout];
    float v = 0.0f;
    if (p.few) {
        const int ci = e / p.k, b = e - ci * p.k;
        if (ci < p.Cin) v = p.w[(((size_t)co * p.Cin + ci) * p.k + tap) * p.k + b];
    } else {
        v = p.w[((size_t)co * p.Cin + e) * p.k * p.k + tap];
    }
    if (p.bf16) static_cast<__nv_bfloat16*>(p.U)[gid] = __float2bfloat16_rn(v);
    else static_cast<float*>(p.U)[gid] = tf32_rn(v);
}

typedef void (*LineKernel)(CUtensorMap, CUtensorMap, LineParams);

template <int KS, bool BF16>
LineKernel line_kernel_of(const LinePlan& p)
{
    auto by_g = [&](auto mt) -> LineKernel {
        constexpr int MT = decltype(mt)::value;
        return p.taps_per_step == 3 ? line_gemm_kernel<MT, KS, 3, BF16> : p.taps_per_step == 2 ? line_gemm_kernel<MT, KS, 2, BF16> : line_gemm_kernel<MT, KS, 1, BF16>;
    };
    return p.mt == 4 ? by_g(std::integral_constant<int, 4>()) : p.mt == 2 ? by_g(std::integral_constant<int, 2>()) : by_g(std::integral_constant<int, 1>());
}

LineKernel line_kernel(const LinePlan& p)
{
    return p.s.bf16 ? line_kernel_of<4, true>(p) : p.k_steps == 4 ? line_kernel_of<4, false>(p) : line_kernel_of<3, false>(p);
}

}  // namespace

cudaError_t line_setup(LineConv* lc, void* A, void* U, const char** why)
{
    lc->ready = false;
    const LinePlan& p = lc->p;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&lc->num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int eb = p.s.bf16 ? 2 : 4;
    if (!encode_operand_map_sw(&lc->map_a, A, eb, p.elems, p.P, p.n_planes, p.P * p.elems, p.box_rows, 128) ||
        !encode_operand_map_sw(&lc->map_u, U, eb, p.elems, p.s.Cout, p.n_taps, (long long)p.s.Cout * p.elems, p.bn, 128)) {
        *why = "cuTensorMapEncodeTiled failed or is unavailable";
        return cudaErrorInvalidValue;
    }
    e = cudaFuncSetAttribute(line_kernel(p), cudaFuncAttributeMaxDynamicSharedMemorySize, kLineSmemBytes);
    if (e != cudaSuccess) return e;
    lc->ready = true;
    return cudaSuccess;
}

cudaError_t launch_line_weights(const LinePlan& lp, const float* w, void* U, cudaStream_t stream)
{
    WeightParams p = {};
    p.w = w;
    p.U = U;
    p.Cout = lp.s.Cout; p.Cin = lp.s.Cin; p.k = lp.s.k; p.elems = lp.elems; p.few = lp.few; p.bf16 = lp.s.bf16; p.n_taps = lp.n_taps;
    for (int i = 0; i < lp.n_taps; ++i) p.tap_id[i] = lp.tap_id[i];
    const long long total = (long long)lp.n_taps * lp.s.Cout * lp.elems;
    line_weights_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_line_pack(const LinePlan& lp, const float* x, void* A, cudaStream_t stream)
{
    PackParams p = {};
    const LineShape& s = lp.s;
    p.x = x;
    p.A = A;
    p.P = lp.P; p.T = lp.T;
    p.Cin = s.Cin; p.H = s.H; p.W = s.W; p.k = s.k; p.stride = s.stride; p.dil = s.dil; p.pad = s.pad; p.strips = lp.strips; p.Hq = lp.Hq; p.Wq = lp.Wq;
    p.elems = lp.elems; p.n_planes = lp.n_planes;
    for (int i = 0; i < lp.n_planes; ++i) {
        p.phase_h[i] = lp.phase_h[i];
        p.phase_w[i] = lp.phase_w[i];
    }
    if (lp.few)
        return launch_overlapped(lp.k_steps == 3 ? line_pack_few_kernel<24> : line_pack_few_kernel<32>, dim3((unsigned)((lp.P + 255) / 256), (unsigned)lp.n_planes),
                                 dim3(256), 0, stream, p);
    const long long gx = (lp.P + 31) / 32 * lp.n_planes;
    if (gx > 2147483647ll || (lp.elems + 63) / 64 > 65535) return cudaErrorInvalidValue;
    return launch_overlapped(s.bf16 ? line_pack_kernel<true> : line_pack_kernel<false>, dim3((unsigned)gx, (unsigned)((lp.elems + 63) / 64)), dim3(256), 0, stream, p);
}

cudaError_t launch_line_gemm(const LineConv& lc, const float* bias, float* y, int relu, int* status, cudaStream_t stream)
{
    if (!lc.ready) return cudaErrorInvalidValue;
    const LinePlan& lp = lc.p;
    LineParams p = {};
    p.bias = bias; p.y = y; p.status = status;
    p.T = lp.T;
    p.n_items = (unsigned)lp.n_items; p.n_tile_blocks = (unsigned)lp.n_tile_blocks;
    p.Cout = lp.s.Cout; p.bn = lp.bn; p.blocks = lp.blocks; p.n_groups = lp.n_groups;
    p.region = lp.region; p.boxes = lp.boxes; p.box_rows = lp.box_rows; p.a_slots = lp.a_slots; p.b_slots = lp.b_slots;
    p.tmem_cols = 32;
    while (p.tmem_cols < 2 * lp.mt * lp.bn) p.tmem_cols *= 2;
    p.strips = lp.strips; p.Hq = lp.Hq; p.Wq = lp.Wq; p.OH = lp.s.OH; p.OW = lp.s.OW; p.relu = relu;
    for (int i = 0; i < lp.n_groups; ++i) {
        p.group_plane[i] = lp.group_plane[i];
        p.group_base[i] = lp.group_base[i];
        p.group_first[i] = lp.group_first[i];
        p.group_taps[i] = lp.group_taps[i];
    }
    for (int i = 0; i < lp.n_taps; ++i) p.tap_rel[i] = lp.tap_rel[i];
    const unsigned grid = lp.n_items < lc.num_sms ? (unsigned)lp.n_items : (unsigned)lc.num_sms;
    // (the full budget: at most one CTA per SM, so that tensor memory is never contended)
    return launch_overlapped(line_kernel(lp), dim3(grid), dim3(line_threads(lp.mt)), (size_t)kLineSmemBytes, stream, lc.map_a, lc.map_u, p);
}

}  // namespace mnnb
