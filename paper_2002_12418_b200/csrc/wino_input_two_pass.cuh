// Winograd input transform V = B^T d B (Eq. 6) as two passes through shared memory.
//
// From alpha = 7 on a tile's alpha x alpha intermediate does not fit the registers beside its arithmetic, and unrolling
// both passes over it makes tens of kilobytes of straight-line code.  Here a warp owns one row of the tiles in the row
// pass and one column in the column pass, so the code is one 1-D transform each (pass_1d of wino_input.cuh) in a short
// loop, on packed pairs of adjacent channels: 16 lanes hold 32 channels of a tile and the warp two tiles.
//
// Work item = (image, tile row, segment of `txs` tiles, block of 32 channels), alpha warps:
//   load:    warp r reads input row r of the segment for the 32 channels (a lane per column, zeros outside the image) and
//            stages it as X [row][column][channel], 34 words per column so that neighbouring columns differ in bank;
//   rows:    warp r transforms row r of every tile, X -> H [row][tile][position][channel];
//   columns: warp j transforms column j of every tile, H -> V, two adjacent channels per lane.
// Two to four persistent CTAs share an SM, and the loads of a CTA's next item are in flight (32 registers per lane) during
// the column pass of this one: with one item per CTA the three phases added up (7 x 7 layer below 92 us instead of 83).
// Rows need no alignment, and an item is short, so small layers spread over many SMs.
//
// Measured, transform only, against the ring kernel in column sweeps: 128 channels 28 x 28 batch 64 with 7 x 7 kernels
// (alpha = 10, TF32 hi + lo) 98 -> 83 us, with 5 x 5 (alpha = 8, BF16 hi + lo) 41 -> 37 us; one image of 64 channels with
// 7 x 7 8.6 -> 5.0 us; 64 channels 45 x 45 batch 4 with 7 x 7 17.3 -> 7.8 us.  3 x 3 kernels (alpha = 6): 64 channels 75 x
// 75 batch 8 20.3 -> 12.9 us, 8 channels 300 x 301 32.1 -> 10.6 us.
#pragma once

#include <algorithm>

#include "wino_input.cuh"

namespace mnnb {
namespace wino {

constexpr int kTpChannels = 32, kTpPitch = 34;
constexpr int kTpSmem = 200 * 1024;          // of all CTAs of an SM
// CTAs of an SM, by registers (threads x at most 96) and by the shared memory that a segment of 32 columns takes
__host__ __device__ constexpr int tp_ctas(int alpha) { return alpha >= 7 ? 2 : alpha >= 5 ? 3 : 4; }
inline int tp_smem(int alpha, int m, int txs) { return 4 * alpha * (((txs - 1) * m + alpha) * kTpPitch + txs * alpha * kTpChannels); }

struct TwoPassItems {
    int txs, nseg, cols, cblocks;            // tiles per segment, segments per tile row, staged columns (at most 32), channel blocks
    long long n_items;                       // below 2^31
};

template <int ALPHA, bool SYM, int MODE>
__global__ void __launch_bounds__(32 * ALPHA, tp_ctas(ALPHA))
input_transform_two_pass_kernel(const float* __restrict__ x, char* V_hi, char* V_lo, WinoGeom g, TwoPassItems it,
                                const __grid_constant__ MatBt2 Bt)
{
    extern __shared__ __align__(16) float s_x[];                       // X, then H
    float* const s_h = s_x + ALPHA * it.cols * kTpPitch;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int half = lane >> 4, cp = 2 * (lane & 15);
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();
    const size_t plane = (size_t)g.H * g.W;
    float v[kTpChannels];                                              // this lane's column of the next item's row `warp`
    auto decode = [&](unsigned b, int& img, int& ty, int& tx0, int& c0) {
        c0 = (int)(b % (unsigned)it.cblocks) * kTpChannels; b /= (unsigned)it.cblocks;
        tx0 = (int)(b % (unsigned)it.nseg) * it.txs; b /= (unsigned)it.nseg;
        ty = (int)(b % (unsigned)g.th);
        img = (int)(b / (unsigned)g.th);
    };
    auto load = [&](unsigned item) {
        int img, ty, tx0, c0;
        decode(item, img, ty, tx0, c0);
        const int ih = ty * g.m - g.pad + warp, iw = tx0 * g.m - g.pad + lane;
        const bool ok = lane < it.cols && ih >= 0 && ih < g.H && iw >= 0 && iw < g.W;
        const float* src = x + ((size_t)img * g.Cin + c0) * plane + (ok ? (size_t)ih * g.W + iw : 0);
        const int n_c = ok ? g.Cin - c0 : 0;
#pragma unroll
        for (int c = 0; c < kTpChannels; ++c) v[c] = c < n_c ? __ldg(src + (size_t)c * plane) : 0.0f;
    };
    auto stage = [&]() {
        if (lane < it.cols) {
            float* dst = s_x + (warp * it.cols + lane) * kTpPitch;
#pragma unroll
            for (int c = 0; c < kTpChannels; c += 2) *reinterpret_cast<float2*>(dst + c) = make_float2(v[c], v[c + 1]);
        }
        __syncwarp();                                                  // the row pass reads the row this warp has staged
    };
    constexpr int eb = (MODE == STORE_BF16 || MODE == STORE_BF16_SPLIT) ? 2 : 4;
    const long long row_step = (long long)g.v_plane * eb * ALPHA;      // from transform position (i, j) to (i + 1, j)
    const unsigned n_items = (unsigned)it.n_items;
    unsigned item = blockIdx.x;
    if (item < n_items) load(item);
    for (; item < n_items; item += gridDim.x) {
        int img, ty, tx0, c0;
        decode(item, img, ty, tx0, c0);
        const int nt = min(it.txs, g.tw - tx0);
        stage();
#pragma unroll 1
        for (int t = half; t < nt; t += 2) {
            const float* px = s_x + (warp * it.cols + t * g.m) * kTpPitch + cp;
            float2 d[ALPHA], o[ALPHA];
#pragma unroll
            for (int j = 0; j < ALPHA; ++j) d[j] = *reinterpret_cast<const float2*>(px + j * kTpPitch);
            pass_1d<ALPHA, SYM>(d, o, Bt);
            float* ph = s_h + ((warp * it.txs + t) * ALPHA) * kTpChannels + cp;
#pragma unroll
            for (int j = 0; j < ALPHA; ++j) *reinterpret_cast<float2*>(ph + j * kTpChannels) = o[j];
        }
        if (item + gridDim.x < n_items) load(item + gridDim.x);     // in flight during the column pass
        __syncthreads();
        if (c0 + cp < g.cin_pad) {                                     // (cin_pad is even: a pair is whole or absent)
#pragma unroll 1
            for (int t = half; t < nt; t += 2) {
                const float* ph = s_h + (t * ALPHA + warp) * kTpChannels + cp;
                float2 d[ALPHA], o[ALPHA];
#pragma unroll
                for (int r = 0; r < ALPHA; ++r) d[r] = *reinterpret_cast<const float2*>(ph + r * it.txs * (ALPHA * kTpChannels));
                pass_1d<ALPHA, SYM>(d, o, Bt);
                const long long tile = ((long long)img * g.th + ty) * g.tw + tx0 + t;
                const long long off = ((long long)warp * g.v_plane + tile * g.cin_pad + c0 + cp) * eb;
                char* hi = V_hi + off;
                char* lo = V_lo + off;
#pragma unroll
                for (int i = 0; i < ALPHA; ++i) {
                    put<MODE>(hi, lo, o[i]);
                    hi += row_step;
                    lo += row_step;
                }
            }
        }
        __syncthreads();                                               // H is free
    }
}

template <int ALPHA>
TwoPassItems plan_two_pass_items(const WinoGeom& g)
{
    TwoPassItems it;
    int txs = g.tw;
    while (txs > 1 && (tp_smem(ALPHA, g.m, txs) > kTpSmem / tp_ctas(ALPHA) || (txs - 1) * g.m + ALPHA > 32)) --txs;
    it.nseg = (g.tw + txs - 1) / txs;
    it.txs = (g.tw + it.nseg - 1) / it.nseg;
    it.cols = (it.txs - 1) * g.m + ALPHA;
    it.cblocks = (g.cin_pad + kTpChannels - 1) / kTpChannels;
    it.n_items = (long long)g.images * g.th * it.nseg * it.cblocks;
    return it;
}

template <int ALPHA>
cudaError_t launch_input_two_pass(const float* x, void* V_hi, void* V_lo, const WinoGeom& g, const TwoPassItems& it, int mode,
                                  bool sym, const MatBt2& bt, int num_sms, cudaStream_t stream)
{
    if (it.n_items > 2147483647ll) return cudaErrorInvalidConfiguration;
    if (it.n_items <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)std::min<long long>(it.n_items, (long long)tp_ctas(ALPHA) * num_sms);
    const size_t smem = (size_t)tp_smem(ALPHA, g.m, it.txs);
    auto launch = [&](auto kern) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTpSmem / tp_ctas(ALPHA));
        if (e != cudaSuccess) return e;
        return launch_overlapped(kern, dim3(grid), dim3(32 * ALPHA), smem, stream, x, static_cast<char*>(V_hi),
                                 static_cast<char*>(V_lo), g, it, bt);
    };
#define MNNB_TP(MODE) return sym ? launch(input_transform_two_pass_kernel<ALPHA, true, MODE>) : launch(input_transform_two_pass_kernel<ALPHA, false, MODE>)
    switch (mode) {
        case STORE_TF32: MNNB_TP(STORE_TF32);
        case STORE_BF16: MNNB_TP(STORE_BF16);
        case STORE_TF32_SPLIT: MNNB_TP(STORE_TF32_SPLIT);
        case STORE_BF16_SPLIT: MNNB_TP(STORE_BF16_SPLIT);
        default: MNNB_TP(STORE_FP32);
    }
#undef MNNB_TP
}

}  // namespace wino
}  // namespace mnnb
