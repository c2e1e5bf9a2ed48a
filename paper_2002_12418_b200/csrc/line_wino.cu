// Row-wise Winograd: V = B^T d along the rows only (wino_rect.cu), a product that sums over the kernel rows as well as the
// channels, y = A^T M along the rows (wino_rect.cu).  Against the two-dimensional form F(m x m, k x k) the product has k m / alpha
// times the multiplications, but V and M are m / alpha as large ((alpha / m) times x and y instead of its square), and one
// axis of rounding error less, which lets large kernels use BF16 hi + lo operands.
//
// Measured, three kernels: 5 x 5 128 channels 28 x 28 batch 64, F(4, 5): 18 + 43 + 20 us against 98 in two dimensions; 7 x 7, F(2, 7):
// 45 + 107 + 31 us against 208 (F(4, 7) takes 126 us for its product, but with an error of 9e-5).  Error against 64 bits over 27 random layers:
// 1.5 to 1.6e-5 (3 x 3), 1.6 to 2.1e-5 (5 x 5), 1.8 to 2.7e-5 (7 x 7), at most 0.36 of the form each replaced.  The product reaches 0.75 of
// the tensor core's time: 128 x 128 x 16 instructions, 75 cycles each.
//
// The product is the persistent pipeline of line_conv.cu over items (position xi, block of tiles, block of channels): a region of
// 128 * mt + (k - 1) * tiles_w consecutive tiles x 32 channels, hi and lo, is staged once per block of channels in the 64-byte
// swizzle and read at k start rows; per kernel row one weight tile, hi and lo; hi*hi + lo*hi + hi*lo into one accumulator.
#include "line_wino.h"

#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "contract_umma.h"
#include "line_plan.h"
#include "umma.cuh"

namespace mnnb {

namespace {

constexpr int kEpiWarps = 8, kThreads = 32 * (2 + kEpiWarps);          // warps 0: copies, 1: MMA
constexpr int kBlock = 32, kRowBytes = 64;                             // channels per stage, bytes of one half of a row
constexpr int kMaxA = 3, kMaxB = 8;
constexpr int kSmemBytes = 208 * 1024;
constexpr int kErrProducer = 81, kErrMmaA = 82, kErrMmaB = 83, kErrMmaAcc = 84, kErrEpilogue = 85;

struct Params {
    float* M;
    int* status;
    long long T, m_row_stride;
    unsigned n_items, n_tile_blocks, n_co_blocks;
    int Cout, bn, blocks, k, tiles_w, rows, boxes, box_rows, a_slots, b_slots, tmem_cols;
};

// High word of the shared-memory descriptors: 8-row groups 512 bytes apart, version, 64-byte swizzle.
constexpr uint32_t kDescHi = (512u >> 4) | (1u << 14) | (4u << 29);

template <int MT>
__global__ void __launch_bounds__(kThreads, 1)
line_wino_kernel(const __grid_constant__ CUtensorMap map_v_hi, const __grid_constant__ CUtensorMap map_v_lo, const __grid_constant__ CUtensorMap map_u_hi,
                 const __grid_constant__ CUtensorMap map_u_lo, const __grid_constant__ Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t a_full[kMaxA], a_empty[kMaxA], b_full[kMaxB], b_empty[kMaxB], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    volatile int* abortp = &abort_flag;

    const int warp = ptx::uniform_warp(), lane = threadIdx.x & 31;
    const uint32_t a_base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t a_half = (uint32_t)p.rows * kRowBytes, b_half = (uint32_t)p.bn * kRowBytes;         // multiples of 512 bytes
    const uint32_t b_base = a_base + (uint32_t)p.a_slots * 2u * a_half;

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.a_slots; ++s) {
            ptx::mbar_init(ptx::smem_u32(&a_full[s]), 1);
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
        ptx::prefetch_tensormap(&map_v_hi);
        ptx::prefetch_tensormap(&map_u_hi);
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

    if (warp == 0) {
        // ------------------------------ regions of V and weight tiles ------------------------------
        uint32_t as = 0, a_phase = 0, bs = 0, b_phase = 0;
        bool ok = true;
        for (unsigned item = blockIdx.x; item < p.n_items && ok; item += gridDim.x) {
            const unsigned r = item / p.n_tile_blocks, tb = item - r * p.n_tile_blocks, xi = r / p.n_co_blocks, nb = r - xi * p.n_co_blocks;
            for (int eb = 0; eb < p.blocks && ok; ++eb) {
                if (!ptx::mbar_wait_warp(ptx::smem_u32(&a_empty[as]), a_phase ^ 1u, abortp)) {
                    ok = false;
                    break;
                }
                if (ptx::elect_one()) {
                    const uint32_t bar = ptx::smem_u32(&a_full[as]), dst = a_base + as * 2u * a_half;
                    ptx::mbar_expect_tx(bar, 2u * a_half);
                    for (int b = 0; b < p.boxes; ++b) {
                        const int row = (int)(tb * 128u * (unsigned)MT) + b * p.box_rows;
                        ptx::tma_load_3d(dst + (uint32_t)(b * p.box_rows) * kRowBytes, &map_v_hi, bar, eb * kBlock, row, (int)xi);
                        ptx::tma_load_3d(dst + a_half + (uint32_t)(b * p.box_rows) * kRowBytes, &map_v_lo, bar, eb * kBlock, row, (int)xi);
                    }
                }
                if (++as == (uint32_t)p.a_slots) {
                    as = 0;
                    a_phase ^= 1u;
                }
                for (int a = 0; a < p.k; ++a) {
                    if (!ptx::mbar_wait_warp(ptx::smem_u32(&b_empty[bs]), b_phase ^ 1u, abortp)) {
                        ok = false;
                        break;
                    }
                    if (ptx::elect_one()) {
                        const uint32_t bar = ptx::smem_u32(&b_full[bs]), dst = b_base + bs * 2u * b_half;
                        ptx::mbar_expect_tx(bar, 2u * b_half);
                        ptx::tma_load_3d(dst, &map_u_hi, bar, eb * kBlock, (int)nb * p.bn, (int)xi * p.k + a);
                        ptx::tma_load_3d(dst + b_half, &map_u_lo, bar, eb * kBlock, (int)nb * p.bn, (int)xi * p.k + a);
                    }
                    if (++bs == (uint32_t)p.b_slots) {
                        bs = 0;
                        b_phase ^= 1u;
                    }
                }
            }
        }
        if (!ok && lane == 0) {
            if (!*abortp) atomicCAS(p.status, 0, kErrProducer);
            *abortp = 1;
        }
    } else if (warp == 1) {
        // ------------------------------ MMA issue ------------------------------
        const uint32_t idesc = ptx::mma_idesc(1, 128, p.bn);
        uint32_t as = 0, a_phase = 0, bs = 0, b_phase = 0, acc = 0, acc_phase = 0;
        int err = 0;
        const uint32_t a_lo0 = (1u << 16) | ((a_base & 0x3FFFFu) >> 4), b_lo0 = (1u << 16) | ((b_base & 0x3FFFFu) >> 4);
        const uint32_t a16 = a_half >> 4, b16 = b_half >> 4;
        for (unsigned item = blockIdx.x; item < p.n_items; item += gridDim.x) {
            if (!ptx::mbar_wait_warp(ptx::smem_u32(&acc_empty[acc]), acc_phase ^ 1u, abortp)) {
                err = kErrMmaAcc;
                goto failed;
            }
            ptx::tc_fence_after();
            const uint32_t d0 = tmem_base + acc * (uint32_t)(MT * p.bn);
            uint32_t accumulate = 0;
            for (int eb = 0; eb < p.blocks; ++eb) {
                if (!ptx::mbar_wait_warp(ptx::smem_u32(&a_full[as]), a_phase, abortp)) {
                    err = kErrMmaA;
                    goto failed;
                }
                for (int t = 0; t < p.k; ++t) {
                    const uint32_t a = a_lo0 + as * 2u * a16 + (uint32_t)(t * p.tiles_w) * (kRowBytes / 16), b = b_lo0 + bs * 2u * b16;
                    if (!ptx::mbar_wait_warp(ptx::smem_u32(&b_full[bs]), b_phase, abortp)) {
                        err = kErrMmaB;
                        goto failed;
                    }
                    if (ptx::elect_one()) {
#pragma unroll
                        for (int pass = 0; pass < 3; ++pass)
#pragma unroll
                            for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                                for (int m = 0; m < MT; ++m)
                                    ptx::mma_lo<1>(d0 + (uint32_t)(m * p.bn), a + (uint32_t)(m * 128 * (kRowBytes / 16) + ks * 2) + (pass == 1 ? a16 : 0u),
                                           b + (uint32_t)(ks * 2) + (pass == 2 ? b16 : 0u), kDescHi, idesc, (pass | ks) ? 1u : accumulate);
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
    } else {
        // ------------------------------ epilogue: store M ------------------------------
        const int q = warp & 3, part = (warp - 2) >> 2;              // tensor-memory lane quarter; which half of the column chunks
        uint32_t acc = 0, acc_phase = 0;
        for (unsigned item = blockIdx.x; item < p.n_items; item += gridDim.x) {
            const unsigned r = item / p.n_tile_blocks, tb = item - r * p.n_tile_blocks, xi = r / p.n_co_blocks, nb = r - xi * p.n_co_blocks;
            int got = 1;
            if (lane == 0) got = ptx::mbar_wait_relaxed(ptx::smem_u32(&acc_full[acc]), acc_phase, abortp) ? 1 : 0;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) {
                if (lane == 0) {
                    if (!*abortp) atomicCAS(p.status, 0, kErrEpilogue);
                    *abortp = 1;
                }
                break;
            }
            ptx::tc_fence_after();
            const int co0 = (int)nb * p.bn, n_co = min(p.bn, p.Cout - co0), n_chunks = (n_co + 15) >> 4;
            for (int m = 0; m < MT; ++m) {
                const long long t = (long long)tb * (128 * MT) + m * 128 + q * 32 + lane;
                const bool live = t < p.T;
                float* const dst = p.M + ((size_t)xi * p.Cout + co0) * p.m_row_stride + (live ? t : 0);
                const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (acc * (uint32_t)MT + (uint32_t)m) * (uint32_t)p.bn;
                auto store = [&](const uint32_t (&v)[16], int ch) {
                    if (!live) return;
                    float* pj = dst + (size_t)(ch * 16) * p.m_row_stride;
                    const int left = n_co - ch * 16;
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        if (e < left) *pj = __uint_as_float(v[e]);
                        pj += p.m_row_stride;
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

struct WeightParams {
    const float* w;
    __nv_bfloat16* U_hi;
    __nv_bfloat16* U_lo;
    int Cout, Cin, cin_pad, k, alpha;
    float G[12 * 7];
};

// A thread per (output channel, input channel), all kernel rows and positions.
__global__ void __launch_bounds__(256) line_wino_weights_kernel(const __grid_constant__ WeightParams p)
{
    const long long gid = (long long)blockIdx.x * 256 + threadIdx.x;
    const long long plane = (long long)p.Cout * p.cin_pad;
    if (gid >= plane) return;
    const int ci = (int)(gid % p.cin_pad), co = (int)(gid / p.cin_pad);
    for (int a = 0; a < p.k; ++a) {
        const float* src = p.w + (((size_t)co * p.Cin + (ci < p.Cin ? ci : 0)) * p.k + a) * p.k;
        for (int xi = 0; xi < p.alpha; ++xi) {
            float s = 0.0f;
            if (ci < p.Cin)
                for (int b = 0; b < p.k; ++b) s = fmaf(p.G[xi * p.k + b], src[b], s);
            const size_t at = (size_t)(xi * p.k + a) * plane + (size_t)gid;
            const __nv_bfloat16 h = __float2bfloat16_rn(s);
            p.U_hi[at] = h;
            p.U_lo[at] = __float2bfloat16_rn(s - __bfloat162float(h));
        }
    }
}

}  // namespace

bool line_wino_plan(const LineWinoShape& s, int num_sms, LineWinoPlan* p)
{
    std::memset(p, 0, sizeof(*p));
    p->s = s;
    auto cdiv = [](long long a, long long b) { return (a + b - 1) / b; };
    auto rup = [&](long long a, long long b) { return cdiv(a, b) * b; };
    p->alpha = s.m + s.k - 1;
    if (p->alpha > 10 || s.k > 7) return false;
    const int reach = s.k - 1;
    p->Hq = axis_pitch(s.OH, s.pad, s.H + s.pad, reach);         // neighbours share their zero rows
    p->tiles_w = (int)cdiv(s.OW, s.m);
    p->T = (long long)s.N * p->Hq * p->tiles_w;
    p->cin_pad = (int)rup(s.Cin, 8);
    p->blocks = (int)cdiv(p->cin_pad, kBlock);
    p->m_row_stride = rup(p->T, 32);
    p->v_bytes = 4 * p->alpha * p->T * p->cin_pad;
    p->u_bytes = 4ll * p->alpha * s.k * s.Cout * p->cin_pad;
    p->m_bytes = 4 * p->alpha * s.Cout * p->m_row_stride;
    if (p->T >= (1ll << 31) - 65536 || p->v_bytes + p->m_bytes > (4ll << 30)) return false;
    const int co16 = (int)rup(s.Cout, 16), span = reach * p->tiles_w;
    long long best = -1;
    for (int mt = 1; mt <= 2; ++mt)
        for (int nb = (int)cdiv(co16, 256); nb <= (int)cdiv(co16, 16) && nb <= 64; ++nb) {
            const int bn = (int)rup(cdiv(co16, nb), 16);
            if (2 * mt * bn > 512) continue;
            const int need = 128 * mt + span, boxes = (int)cdiv(need, 256), box_rows = (int)rup(cdiv(need, boxes), 8), rows = boxes * box_rows;
            const long long a_slot = 2ll * rows * kRowBytes, b_slot = 2ll * bn * kRowBytes, room = kSmemBytes - 1024;
            if (2 * a_slot + 3 * b_slot > room) continue;
            const int b_slots = (int)std::min<long long>(kMaxB, (room - 2 * a_slot) / b_slot);
            const int a_slots = (int)std::min<long long>(kMaxA, (room - b_slots * b_slot) / a_slot);
            const long long tile_blocks = cdiv(p->T, 128 * mt), items = tile_blocks * nb * p->alpha;
            if (items >= (1ll << 31)) continue;
            // an item: six instructions per kernel row and block of channels (57 cycles for the left operand, more only from 128
            // channels on), or the delivery of its operands; or its drain
            const long long mma = 6ll * mt * s.k * std::max(bn / 2, 57 + bn / 7) * 555, load = (a_slot + s.k * b_slot) * 63 / 5;
            const long long drain = (long long)mt * bn * 512 * 28 + 1087000, loop = p->blocks * std::max(mma, load) + 285000;
            const long long cost = cdiv(items, num_sms) * std::max(loop, drain) + drain;
            if (best >= 0 && cost >= best) continue;
            best = cost;
            p->mt = mt; p->bn = bn; p->n_co_blocks = nb; p->rows = rows; p->boxes = boxes; p->box_rows = box_rows;
            p->a_slots = a_slots; p->b_slots = b_slots; p->n_tile_blocks = tile_blocks; p->n_items = items; p->product_ps = cost;
        }
    p->tmem_cols = 32;
    while (p->tmem_cols < 2 * p->mt * p->bn) p->tmem_cols *= 2;
    return best >= 0;
}

cudaError_t line_wino_setup(LineWino* lw, void* V, void* U, const char** why)
{
    lw->ready = false;
    const LineWinoPlan& p = lw->p;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&lw->num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    char *v_lo = static_cast<char*>(V) + p.v_bytes / 2, *u_lo = static_cast<char*>(U) + p.u_bytes / 2;
    const long long u_planes = (long long)p.alpha * p.s.k, u_plane = (long long)p.s.Cout * p.cin_pad, v_plane = p.T * p.cin_pad;
    if (!encode_operand_map_sw(&lw->map_v_hi, V, 2, p.cin_pad, p.T, p.alpha, v_plane, p.box_rows, kRowBytes) ||
        !encode_operand_map_sw(&lw->map_v_lo, v_lo, 2, p.cin_pad, p.T, p.alpha, v_plane, p.box_rows, kRowBytes) ||
        !encode_operand_map_sw(&lw->map_u_hi, U, 2, p.cin_pad, p.s.Cout, u_planes, u_plane, p.bn, kRowBytes) ||
        !encode_operand_map_sw(&lw->map_u_lo, u_lo, 2, p.cin_pad, p.s.Cout, u_planes, u_plane, p.bn, kRowBytes)) {
        *why = "cuTensorMapEncodeTiled failed or is unavailable";
        return cudaErrorInvalidValue;
    }
    e = cudaFuncSetAttribute(p.mt == 2 ? line_wino_kernel<2> : line_wino_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    lw->ready = e == cudaSuccess;
    return e;
}

cudaError_t launch_line_wino_weights(const LineWinoPlan& lp, const float* w, void* U, const float* G, cudaStream_t stream)
{
    WeightParams p = {};
    p.w = w;
    p.U_hi = static_cast<__nv_bfloat16*>(U);
    p.U_lo = reinterpret_cast<__nv_bfloat16*>(static_cast<char*>(U) + lp.u_bytes / 2);
    p.Cout = lp.s.Cout; p.Cin = lp.s.Cin; p.cin_pad = lp.cin_pad; p.k = lp.s.k; p.alpha = lp.alpha;
    for (int i = 0; i < lp.alpha * lp.s.k; ++i) p.G[i] = G[i];
    const long long total = (long long)lp.s.Cout * lp.cin_pad;
    line_wino_weights_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_line_wino_product(const LineWino& lw, float* M, int* status, cudaStream_t stream)
{
    if (!lw.ready) return cudaErrorInvalidValue;
    const LineWinoPlan& lp = lw.p;
    Params p = {};
    p.M = M; p.status = status;
    p.T = lp.T; p.m_row_stride = lp.m_row_stride;
    p.n_items = (unsigned)lp.n_items; p.n_tile_blocks = (unsigned)lp.n_tile_blocks; p.n_co_blocks = (unsigned)lp.n_co_blocks;
    p.Cout = lp.s.Cout; p.bn = lp.bn; p.blocks = lp.blocks; p.k = lp.s.k; p.tiles_w = lp.tiles_w; p.rows = lp.rows; p.boxes = lp.boxes; p.box_rows = lp.box_rows;
    p.a_slots = lp.a_slots; p.b_slots = lp.b_slots; p.tmem_cols = lp.tmem_cols;
    const unsigned grid = lp.n_items < lw.num_sms ? (unsigned)lp.n_items : (unsigned)lw.num_sms;
    // (the full budget: at most one CTA per SM, so that tensor memory is never contended)
    return launch_overlapped(lp.mt == 2 ? line_wino_kernel<2> : line_wino_kernel<1>, dim3(grid), dim3(kThreads), (size_t)kSmemBytes, stream, lw.map_v_hi, lw.map_v_lo,
                             lw.map_u_hi, lw.map_u_lo, p);
}

}  // namespace mnnb
