// Templates of the Winograd input and output transform kernels; instantiated per
// alpha in wino_inst_*.cu so that the translation units compile in parallel.
#pragma once
#include <cuda_bf16.h>

#include <algorithm>

#include "kernels.h"
#include "wino_input_two_pass.cuh"

namespace mnnb {
namespace wino {

struct MatBt { float v[12 * 12]; };
struct MatAt { float v[6 * 12]; };
struct MatG { float v[12 * 7]; };

__device__ __forceinline__ float round_tf32(float v)
{
    uint32_t u;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(v));
    return __uint_as_float(u);
}

// Store one transformed value in the operand format(s).
__device__ __forceinline__ void store_operand(void* hi, void* lo, size_t idx, float v, int mode)
{
    switch (mode) {
        case STORE_TF32:
            reinterpret_cast<float*>(hi)[idx] = round_tf32(v);
            break;
        case STORE_BF16:
            reinterpret_cast<__nv_bfloat16*>(hi)[idx] = __float2bfloat16_rn(v);
            break;
        case STORE_TF32_SPLIT: {
            const float h = round_tf32(v);
            reinterpret_cast<float*>(hi)[idx] = h;
            reinterpret_cast<float*>(lo)[idx] = round_tf32(v - h);
            break;
        }
        case STORE_BF16_SPLIT: {
            const __nv_bfloat16 h = __float2bfloat16_rn(v);
            reinterpret_cast<__nv_bfloat16*>(hi)[idx] = h;
            reinterpret_cast<__nv_bfloat16*>(lo)[idx] = __float2bfloat16_rn(v - __bfloat162float(h));
            break;
        }
        default:
            reinterpret_cast<float*>(hi)[idx] = v;
            break;
    }
}

// ---------------------------------------------------------------------------
// Output transform: one thread per (tile, output channel); consecutive threads
// take consecutive tiles, so the alpha^2 reads of M[xi][co][tile] are coalesced
// and the m-wide row pieces written to y are adjacent in memory.
// ---------------------------------------------------------------------------
constexpr int kOutThreads = 128;

template <int ALPHA, int M>
__global__ void __launch_bounds__(kOutThreads) output_transform_kernel(const float* __restrict__ Mx,
                                                                       const float* __restrict__ bias,
                                                                       float* __restrict__ y, WinoGeom g, int relu, MatAt At)
{
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();
    const long long tile = (long long)blockIdx.x * kOutThreads + threadIdx.x;
    const int co = blockIdx.y;
    if (tile >= g.tiles) return;
    float acc[ALPHA][ALPHA];
    const float* src = Mx + (size_t)co * g.m_row_stride + tile;
    const size_t plane = (size_t)g.Cout * g.m_row_stride;
#pragma unroll
    for (int i = 0; i < ALPHA; ++i)
#pragma unroll
        for (int j = 0; j < ALPHA; ++j) acc[i][j] = __ldcs(src + (size_t)(i * ALPHA + j) * plane);

    float t[M][ALPHA];
#pragma unroll
    for (int a = 0; a < M; ++a)
#pragma unroll
        for (int j = 0; j < ALPHA; ++j) {
            float s = 0.0f;
#pragma unroll
            for (int i = 0; i < ALPHA; ++i) s = fmaf(At.v[a * ALPHA + i], acc[i][j], s);
            t[a][j] = s;
        }
    const int tx = (int)(tile % g.tw);
    const long long rest = tile / g.tw;
    const int ty = (int)(rest % g.th);
    const int img = (int)(rest / g.th);
    const float b = bias ? __ldg(bias + co) : 0.0f;
    float* dst = y + (((size_t)img * g.Cout + co) * g.OH + (size_t)ty * M) * g.OW + (size_t)tx * M;
    const int rows = min(M, g.OH - ty * M), cols = min(M, g.OW - tx * M);
#pragma unroll
    for (int a = 0; a < M; ++a) {
        float o[M];
#pragma unroll
        for (int c = 0; c < M; ++c) {
            float s = b;
#pragma unroll
            for (int j = 0; j < ALPHA; ++j) s = fmaf(t[a][j], At.v[c * ALPHA + j], s);
            o[c] = relu ? fmaxf(s, 0.0f) : s;
        }
        if (a < rows) {
            float* row = dst + (size_t)a * g.OW;
            if (cols == M && (M % 2 == 0) && ((reinterpret_cast<uintptr_t>(row) & 7u) == 0)) {
#pragma unroll
                for (int c = 0; c < M; c += 2) *reinterpret_cast<float2*>(row + c) = make_float2(o[c], o[c + 1]);
            } else {
#pragma unroll
                for (int c = 0; c < M; ++c)
                    if (c < cols) row[c] = o[c];
            }
        }
    }
}

template <int ALPHA, int M>
cudaError_t launch_output_am(const float* Mx, const float* bias, float* y, const WinoGeom& g, int relu,
                             const TransformMatrices& mats, cudaStream_t stream)
{
    MatAt at;
    for (int i = 0; i < M * ALPHA; ++i) at.v[i] = mats.At[i];
    dim3 grid((unsigned)((g.tiles + kOutThreads - 1) / kOutThreads), (unsigned)g.Cout);
    return launch_overlapped(output_transform_kernel<ALPHA, M>, grid, dim3(kOutThreads), 0, stream, Mx, bias, y, g, relu, at);
}

// Defined beside the other tensor-map code (contract_umma.cu).
bool encode_input_map(CUtensorMap* map, const float* x, int images, int C, int H, int W, int box_w);

// Input transform.  Which kernel, by tile, alignment and size (whole layers, us):
//   alpha >= 7               two-pass: the ring kernel would have to sweep the tile in parts.
//   rows that TMA can address (W a multiple of 4, Cin even)
//                            ring; but from alpha = 5 on two-pass where its CTAs fit the chip at once, since it
//                            has no pipeline to fill: 128 channels 28 x 28 batch 1 / 8 / 12 / 16, alpha = 6: 12.5 / 17.2 /
//                            21.1 / 21.1 ring, 12.2 / 15.1 / 18.8 / 20.5 two-pass (224 / 336 / 448 CTAs of 444); beyond, 64
//                            channels 56 x 56 batch 32 52 / 61.  alpha = 4: 64 channels 56 x 56 11.4 / 12.9.
//   other rows               two-pass; but the plane kernel up to 16 columns where two-pass CTAs come more than once to a
//                            slot: 512 channels 7 x 7 batch 8 / 16 / 32 17.0 / 19.5 / 24.6 plane, 15.0 / 18.9 / 26.5 two-pass.
template <int ALPHA>
cudaError_t launch_input(const float* x, void* V_hi, void* V_lo, const WinoGeom& g, int mode, const TransformMatrices& mats,
                         int* status, int num_sms, cudaStream_t stream)
{
    MatBt2 bt;
    for (int i = 0; i < ALPHA * ALPHA; ++i) bt.v[i] = make_float2(mats.Bt[i], mats.Bt[i]);
    const bool sym = bt_has_symmetric_structure(mats.Bt, ALPHA);
    const TwoPassItems tp = plan_two_pass_items<ALPHA>(g);
    if constexpr (ALPHA <= 6) {
        const bool one_wave = tp.n_items <= (long long)tp_ctas(ALPHA) * num_sms;
        const bool tma_ok = g.W % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15u) == 0 && g.Cin % 2 == 0;
        InputItems it;
        PlaneItems pi;
        size_t smem = 0;
        CUtensorMap xmap;
        auto launch = [&](auto kern, unsigned blocks, unsigned threads, auto&&... args) -> cudaError_t {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kItSmemBudget);
            if (e != cudaSuccess) return e;
            return launch_overlapped(kern, dim3(blocks), dim3(threads), smem, stream, x, args...);
        };
        if (tma_ok) {
            if (!(one_wave && ALPHA >= 5) && plan_input_items(g, ALPHA, num_sms, &it) &&
                encode_input_map(&xmap, x, g.images, g.Cin, g.H, g.W, it.wb)) {
                smem = (size_t)it.nbuf * it.buf_words * sizeof(float);
                const unsigned blocks = (unsigned)std::min<long long>(it.n_items, num_sms);
                if (blocks == 0) return cudaSuccess;
                return launch(sym ? input_transform_ws_kernel<ALPHA, true> : input_transform_ws_kernel<ALPHA, false>, blocks, kItThreads,
                              xmap, static_cast<char*>(V_hi), static_cast<char*>(V_lo), g, it, mode, bt, status);
            }
        } else if (!one_wave && plan_plane_items(g, ALPHA, num_sms, &pi, &smem)) {
            // half the threads where several CTAs come to an SM: two then share it (the registers allow 512 threads)
            const unsigned blocks = (unsigned)(g.images * pi.bands * pi.cblocks);
            const unsigned threads = smem <= kItSmemBudget / 2 && blocks > (unsigned)num_sms ? kItThreads / 2 : kItThreads;
            return launch(sym ? input_transform_plane_kernel<ALPHA, true> : input_transform_plane_kernel<ALPHA, false>, blocks, threads,
                          static_cast<char*>(V_hi), static_cast<char*>(V_lo), g, pi, mode, bt);
        }
    }
    return launch_input_two_pass<ALPHA>(x, V_hi, V_lo, g, tp, mode, sym, bt, num_sms, stream);
}

}  // namespace wino
}  // namespace mnnb

// One non-template entry point per instantiation, defined in wino_inst_*.cu.
#define MNNB_INPUT_FN(A) launch_input_transform_a##A
#define MNNB_OUTPUT_FN(A, MM) launch_output_transform_a##A##_m##MM
#define MNNB_INPUT_ARGS const float *x, void *V_hi, void *V_lo, const WinoGeom &g, int mode, const TransformMatrices &mats, int *status, int num_sms, cudaStream_t stream
#define MNNB_OUTPUT_ARGS const float *Mx, const float *bias, float *y, const WinoGeom &g, int relu, const TransformMatrices &mats, cudaStream_t stream
#define MNNB_DEFINE_INPUT(A) \
    namespace mnnb { cudaError_t MNNB_INPUT_FN(A)(MNNB_INPUT_ARGS) { return wino::launch_input<A>(x, V_hi, V_lo, g, mode, mats, status, num_sms, stream); } }
#define MNNB_DEFINE_OUTPUT(A, MM) \
    namespace mnnb { cudaError_t MNNB_OUTPUT_FN(A, MM)(MNNB_OUTPUT_ARGS) { return wino::launch_output_am<A, MM>(Mx, bias, y, g, relu, mats, stream); } }
#define MNNB_DECLARE_INPUT(A) namespace mnnb { cudaError_t MNNB_INPUT_FN(A)(MNNB_INPUT_ARGS); }
#define MNNB_DECLARE_OUTPUT(A, MM) namespace mnnb { cudaError_t MNNB_OUTPUT_FN(A, MM)(MNNB_OUTPUT_ARGS); }
