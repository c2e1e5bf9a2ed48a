// One-dimensional Winograd F(m, k) for 1 x k and k x 1 kernels (Section 4.2; Eq. 6 along one axis).
#include "wino_rect.h"

#include <cuda_bf16.h>

#include "wino_transforms.cuh"

namespace mnnb {

namespace {

using wino::store_operand;

struct RectMats {
    float Bt[kRectMaxAlpha * kRectMaxAlpha];
    float At[6 * kRectMaxAlpha];
    float G[kRectMaxAlpha * 7];
};

__global__ void rect_weights_kernel(const float* __restrict__ w, void* U_hi, void* U_lo, RectGeom g, int mode, RectMats mt)
{
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long plane = (long long)g.Cout * g.cin_pad;
    if (gid >= plane) return;
    const int ci = (int)(gid % g.cin_pad), co = (int)(gid / g.cin_pad);
    float tap[7];
    for (int a = 0; a < g.k; ++a) tap[a] = ci < g.Cin ? w[((size_t)co * g.Cin + ci) * g.k + a] : 0.0f;
    for (int xi = 0; xi < g.alpha; ++xi) {
        float s = 0.0f;
        for (int a = 0; a < g.k; ++a) s = fmaf(mt.G[xi * g.k + a], tap[a], s);
        store_operand(U_hi, U_lo, (size_t)xi * plane + (size_t)gid, s, mode);
    }
}

// The line a tile lies on and its first input position along the long axis.
struct RectTile {
    int n, fixed, start;                 // image; input row (along_w) or input column; first position
};
__device__ __forceinline__ RectTile rect_tile(const RectGeom& g, long long t)
{
    RectTile r;
    if (g.along_w) {
        const int seg = (int)(t % g.n_seg);
        const long long q = t / g.n_seg;
        r.fixed = (int)(q % g.lines) - g.pad_h;
        r.n = (int)(q / g.lines);
        r.start = seg * g.m - g.pad_w;
    } else {
        r.fixed = (int)(t % g.OW) - g.pad_w;
        const long long q = t / g.OW;
        r.n = (int)(q / g.n_seg);
        r.start = (int)(q % g.n_seg) * g.m - g.pad_h;
    }
    return r;
}

// V = B^T d along the long axis.  A CTA holds 16 tiles x 64 channels: lanes run over tiles while x is read (the alpha inputs of
// neighbouring tiles overlap, so all but the first touch of a sector hits L1), and a lane writes two adjacent channels of
// a tile, 128 or 256 bytes of a row of V per warp, after a transposition through shared memory (channel c in row
// (c & 1) * 32 + c / 2 of 17 words: both sides free of bank conflicts).  Bound by the L1 requests of the loads.  Alpha and
// the operand format are compile-time constants and the launch overlaps the previous kernel's end: 192 channels 17 x 17
// batch 32, 1 x 7: 24.0 -> 10.8 us.
constexpr int kRectTiles = 16, kRectChannels = 64;

// VEC: the padding that keeps the size, tiles of VEC outputs and rows of a multiple of VEC columns: a tile's window lies in three
// aligned 128-bit pieces (VEC = 4, k = alpha - 3) or five 64-bit ones (VEC = 2, 7 x 7).  5 x 5 128 channels 28 x 28 batch 64 18 us,
// 64 channels 56 x 56 batch 32 3 x 3 13 us.
template <int ALPHA, int MODE, int VEC>
__global__ void __launch_bounds__(256) rect_input_kernel(const float* __restrict__ x, void* V_hi, void* V_lo, RectGeom g,
                                                         const __grid_constant__ RectMats mt)
{
    __shared__ float s[ALPHA][kRectChannels][kRectTiles + 1];
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();
    const long long t0 = (long long)blockIdx.x * kRectTiles;
    const int c0 = blockIdx.y * kRectChannels;
    {
        const int tl = threadIdx.x & 15;
        const long long t = t0 + tl;
        const bool t_ok = t < g.tiles;
        const RectTile r = rect_tile(g, t_ok ? t : 0);
        const int fixed_extent = g.along_w ? g.H : g.W, long_extent = g.along_w ? g.W : g.H, step = g.along_w ? 1 : g.W;
        const bool line_ok = t_ok && r.fixed >= 0 && r.fixed < fixed_extent;
        unsigned mask = 0;
#pragma unroll
        for (int j = 0; j < ALPHA; ++j)
            if (line_ok && r.start + j >= 0 && r.start + j < long_extent) mask |= 1u << j;
        const size_t plane = (size_t)g.H * g.W;
        const float* base = x + (size_t)r.n * g.Cin * plane + (g.along_w ? (ptrdiff_t)r.fixed * g.W + r.start : (ptrdiff_t)r.start * g.W + r.fixed);
#pragma unroll 2
        for (int cl = threadIdx.x >> 4; cl < kRectChannels; cl += 16) {
            const int c = c0 + cl;
            const float* src = base + (size_t)(c < g.Cin ? c : 0) * plane;
            float d[ALPHA];
            if constexpr (VEC == 2) {
                static_assert(ALPHA == 8 || VEC != 2, "7 x 7");
                float f[10];
#pragma unroll
                for (int q = 0; q < 5; ++q) {                        // columns start - 1 + 2 q, a pair of them inside the row or outside
                    const int at = r.start - 1 + 2 * q;
                    const float2 v = line_ok && c < g.Cin && at >= 0 && at < g.W ? __ldg(reinterpret_cast<const float2*>(src - 1 + 2 * q)) : make_float2(0.0f, 0.0f);
                    f[2 * q] = v.x;
                    f[2 * q + 1] = v.y;
                }
#pragma unroll
                for (int j = 0; j < ALPHA; ++j) d[j] = f[1 + (j < 9 ? j : 0)];
            } else if constexpr (VEC == 4) {
                constexpr int OFF = 4 - (ALPHA - 4) / 2;             // the window starts here in the first piece
                float f[12];
                const float4* piece = reinterpret_cast<const float4*>(src - OFF);
                const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                const bool in = line_ok && c < g.Cin;
                const float4 q0 = in && r.start > 0 ? __ldg(piece) : zero, q1 = in ? __ldg(piece + 1) : zero,
                             q2 = in && r.start - OFF + 8 < g.W ? __ldg(piece + 2) : zero;
                f[0] = q0.x; f[1] = q0.y; f[2] = q0.z; f[3] = q0.w;
                f[4] = q1.x; f[5] = q1.y; f[6] = q1.z; f[7] = q1.w;
                f[8] = q2.x; f[9] = q2.y; f[10] = q2.z; f[11] = q2.w;
#pragma unroll
                for (int j = 0; j < ALPHA; ++j) d[j] = f[OFF + j];
            } else {
#pragma unroll
                for (int j = 0; j < ALPHA; ++j) d[j] = ((mask >> j) & 1u) && c < g.Cin ? __ldg(src + j * step) : 0.0f;
            }
            float* dst = &s[0][(cl & 1) * 32 + (cl >> 1)][tl];
#pragma unroll
            for (int xi = 0; xi < ALPHA; ++xi) {
                float v = mt.Bt[xi * ALPHA] * d[0];
#pragma unroll
                for (int j = 1; j < ALPHA; ++j) v = fmaf(mt.Bt[xi * ALPHA + j], d[j], v);
                dst[xi * (kRectChannels * (kRectTiles + 1))] = v;
            }
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = c0 + 2 * lane;
    if (c >= g.cin_pad) return;          // (cin_pad is a multiple of 8, so a pair is whole or absent)
    constexpr int eb = (MODE == STORE_BF16 || MODE == STORE_BF16_SPLIT) ? 2 : 4;
    const size_t plane = (size_t)g.tiles * g.cin_pad;
#pragma unroll 4
    for (int q = warp; q < ALPHA * kRectTiles; q += 8) {
        const int xi = q / kRectTiles, tl = q - xi * kRectTiles;
        if (t0 + tl >= g.tiles) continue;
        const size_t off = (xi * plane + (size_t)(t0 + tl) * g.cin_pad + c) * eb;
        wino::put<MODE>(static_cast<char*>(V_hi) + off, static_cast<char*>(V_lo) + off, make_float2(s[xi][lane][tl], s[xi][32 + lane][tl]));
    }
}

template <int ALPHA, int M>
__global__ void __launch_bounds__(128) rect_output_kernel(const float* __restrict__ Mx, const float* __restrict__ bias,
                                                          float* __restrict__ y, RectGeom g, int relu, const __grid_constant__ RectMats mt)
{
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int co = blockIdx.y;
    if (t >= g.tiles) return;
    const size_t plane = (size_t)g.Cout * g.m_row_stride;
    const float* src = Mx + (size_t)co * g.m_row_stride + t;
    float mv[ALPHA];
#pragma unroll
    for (int xi = 0; xi < ALPHA; ++xi) mv[xi] = __ldcs(src + xi * plane);
    const float b = bias ? __ldg(bias + co) : 0.0f;
    int n, oh, ow, step, limit;
    if (g.along_w) {
        const int seg = (int)(t % g.n_seg);
        const long long r = t / g.n_seg;
        oh = (int)(r % g.lines);
        n = (int)(r / g.lines);
        if (oh >= g.OH) return;
        ow = seg * M;
        step = 1;
        limit = g.OW - ow;
    } else {
        ow = (int)(t % g.OW);
        const long long r = t / g.OW;
        n = (int)(r / g.n_seg);
        oh = (int)(r % g.n_seg) * M;
        step = g.OW;
        limit = g.OH - oh;
    }
    float* dst = y + (((size_t)n * g.Cout + co) * g.OH + oh) * g.OW + ow;
#pragma unroll
    for (int a = 0; a < M; ++a) {
        float v = b;
#pragma unroll
        for (int xi = 0; xi < ALPHA; ++xi) v = fmaf(mt.At[a * ALPHA + xi], mv[xi], v);
        if (a < limit) dst[(size_t)a * step] = relu ? fmaxf(v, 0.0f) : v;
    }
}

RectMats pack(const TransformMatrices& mats, const RectGeom& g)
{
    RectMats mt = {};
    for (int i = 0; i < g.alpha * g.alpha; ++i) mt.Bt[i] = mats.Bt[i];
    for (int i = 0; i < g.m * g.alpha; ++i) mt.At[i] = mats.At[i];
    for (int i = 0; i < g.alpha * g.k; ++i) mt.G[i] = mats.G[i];
    return mt;
}

bool geom_ok(const RectGeom& g) { return g.alpha <= kRectMaxAlpha && g.alpha == g.m + g.k - 1 && g.k <= 7 && g.m <= 6; }

}  // namespace

cudaError_t launch_rect_weights(const float* w, void* U_hi, void* U_lo, const RectGeom& g, int mode, const TransformMatrices& mats,
                                cudaStream_t stream)
{
    if (!geom_ok(g)) return cudaErrorInvalidValue;
    const long long total = (long long)g.Cout * g.cin_pad;
    rect_weights_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(w, U_hi, U_lo, g, mode, pack(mats, g));
    return cudaGetLastError();
}

namespace {

template <int ALPHA>
cudaError_t launch_rect_input_alpha(const float* x, void* V_hi, void* V_lo, const RectGeom& g, int mode, const RectMats& mt, dim3 grid,
                                    cudaStream_t stream)
{
    auto kern = mode == STORE_TF32 ? rect_input_kernel<ALPHA, STORE_TF32, 1>
                : mode == STORE_BF16 ? rect_input_kernel<ALPHA, STORE_BF16, 1>
                : mode == STORE_TF32_SPLIT ? rect_input_kernel<ALPHA, STORE_TF32_SPLIT, 1> : rect_input_kernel<ALPHA, STORE_BF16_SPLIT, 1>;
    if constexpr (ALPHA == 6 || ALPHA == 8 || ALPHA == 10)
        if (mode == STORE_BF16_SPLIT && g.along_w && g.m == 4 && g.W % 4 == 0 && g.pad_w == (ALPHA - 4) / 2) kern = rect_input_kernel<ALPHA, STORE_BF16_SPLIT, 4>;
    if constexpr (ALPHA == 8)
        if (mode == STORE_BF16_SPLIT && g.along_w && g.m == 2 && g.W % 2 == 0 && g.pad_w == 3) kern = rect_input_kernel<ALPHA, STORE_BF16_SPLIT, 2>;
    return launch_overlapped(kern, grid, dim3(256), 0, stream, x, V_hi, V_lo, g, mt);
}

}  // namespace

cudaError_t launch_rect_input(const float* x, void* V_hi, void* V_lo, const RectGeom& g, int mode, const TransformMatrices& mats,
                              cudaStream_t stream)
{
    const long long gx = (g.tiles + kRectTiles - 1) / kRectTiles;
    const int gy = (g.cin_pad + kRectChannels - 1) / kRectChannels;
    if (!geom_ok(g) || gx > 2147483647ll || gy > 65535 || mode == STORE_FP32) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)gx, (unsigned)gy);
    const RectMats mt = pack(mats, g);
    switch (g.alpha) {
        case 3: return launch_rect_input_alpha<3>(x, V_hi, V_lo, g, mode, mt, grid, stream);
        case 4: return launch_rect_input_alpha<4>(x, V_hi, V_lo, g, mode, mt, grid, stream);
        case 5: return launch_rect_input_alpha<5>(x, V_hi, V_lo, g, mode, mt, grid, stream);
        case 6: return launch_rect_input_alpha<6>(x, V_hi, V_lo, g, mode, mt, grid, stream);
        case 7: return launch_rect_input_alpha<7>(x, V_hi, V_lo, g, mode, mt, grid, stream);
        case 8: return launch_rect_input_alpha<8>(x, V_hi, V_lo, g, mode, mt, grid, stream);
        case 10: return launch_rect_input_alpha<10>(x, V_hi, V_lo, g, mode, mt, grid, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_rect_output(const float* M, const float* bias, float* y, const RectGeom& g, int relu, const TransformMatrices& mats,
                               cudaStream_t stream)
{
    if (!geom_ok(g) || g.Cout > 65535) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)((g.tiles + 127) / 128), (unsigned)g.Cout);
    const RectMats mt = pack(mats, g);
#define MNNB_RECT_OUT(A, MM) \
    if (g.alpha == A && g.m == MM) return launch_overlapped(rect_output_kernel<A, MM>, grid, dim3(128), 0, stream, M, bias, y, g, relu, mt);
    MNNB_RECT_OUT(3, 2) MNNB_RECT_OUT(5, 4) MNNB_RECT_OUT(7, 6)       // k = 2
    MNNB_RECT_OUT(4, 2) MNNB_RECT_OUT(6, 4) MNNB_RECT_OUT(8, 6)       // k = 3
    MNNB_RECT_OUT(6, 2) MNNB_RECT_OUT(8, 4) MNNB_RECT_OUT(10, 6)      // k = 5
    MNNB_RECT_OUT(8, 2) MNNB_RECT_OUT(10, 4)                          // k = 7
#undef MNNB_RECT_OUT
    return cudaErrorInvalidValue;
}

}  // namespace mnnb
