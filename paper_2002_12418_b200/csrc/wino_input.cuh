// Winograd input transform V = B^T d B (Eq. 6): 1-D passes, operand stores, and two of its three kernels.
//
// The ring kernel (tiles up to alpha = 6, rows aligned for TMA) is persistent and warp-specialised.  Work item = (image,
// tile row, segment of up to `txs` tiles of that row, block of 64 channels).  The alpha input rows of an item are staged
// in a ring of shared-memory buffers laid out [row][channel slot][column]; the number of staged columns `wb` is an odd
// multiple of 4 words, so that 32 lanes reading 128-bit vectors from 32 consecutive slots touch every bank once.  One
// loader warp issues TMA box copies, two per input row (32 channels each, even and odd, through a 5-D view of x that
// splits the channel parity); everything outside the image, including the zero padding of the convolution and channels
// beyond Cin, arrives as zeros, so several items are in flight with no load instructions at all.  The remaining warps
// take (item, tile) units in order.  A lane transforms one tile of TWO adjacent channels held as packed fp32 pairs
// (packed fp32x2 multiply-adds) and writes one 128- or 256-byte row piece of V[xi][tile][channel] per warp store.
//
// Which kernel runs (launch_input): larger tiles, rows that TMA cannot address, and layers that fill the chip at most once
// take the two-pass kernel (wino_input_two_pass.cuh); narrow unaligned planes the kernel at the end of this file.
//
// When the interpolation points are symmetric (0, +-p1, +-p2, ..., infinity; alpha even)
// B^T has a fixed zero pattern and its +p / -p rows share coefficients up to sign
// (the generator polynomial of Eq. 8 is odd), so each 1-D pass needs about half the
// multiplies of the dense form.  The host checks the pattern on the generated matrix
// and otherwise selects the dense form.
//
// Loader and compute warps hand buffers over through mbarriers; every wait is bounded
// and reports through the plan's status word instead of hanging.
#pragma once
#include <cuda_bf16.h>

#include <algorithm>

#include "kernels.h"
#include "umma.cuh"

namespace mnnb {
namespace wino {

constexpr int kItChannels = 64;         // channels per work item
constexpr int kItWarps = 16;
constexpr int kItThreads = 32 * kItWarps;
constexpr int kItMaxBuffers = 6;
constexpr int kItSmemBudget = 200 * 1024;
constexpr int kErrInputLoaderWait = 11, kErrInputComputeWait = 12;

struct MatBt2 { float2 v[12 * 12]; };   // B^T with every entry duplicated into a pair

struct InputItems {
    int txs;            // tiles per item
    int nseg;           // segments per tile row
    int wb;             // staged columns per channel row: 4 x odd words
    int nbuf;           // ring depth
    int cblocks;        // blocks of 64 channels
    int buf_words;      // words per buffer = alpha * 64 * wb
    long long n_items;
};

__device__ __forceinline__ float round_tf32_v(float v)
{
    uint32_t u;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(v));
    return __uint_as_float(u);
}

// ---- two adjacent channels per lane ----
__device__ __forceinline__ float2 v_mul(float2 c, float2 a) { return __fmul2_rn(c, a); }
__device__ __forceinline__ float2 v_fma(float2 c, float2 a, float2 acc) { return __ffma2_rn(c, a, acc); }
__device__ __forceinline__ float2 v_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 v_sub(float2 a, float2 b) { return __ffma2_rn(make_float2(-1.0f, -1.0f), b, a); }

// One 1-D pass o = B^T d.  SYM: the symmetric-point structure described above.
template <int ALPHA, bool SYM>
__device__ __forceinline__ void pass_1d(const float2 (&d)[ALPHA], float2 (&o)[ALPHA], const MatBt2& Bt)
{
    if (SYM) {
        {
            // row of the point 0: even powers only
            float2 s = v_mul(Bt.v[0], d[0]);
#pragma unroll
            for (int r = 2; r < ALPHA; r += 2) s = v_fma(Bt.v[r], d[r], s);
            o[0] = s;
        }
        {
            // row of the point at infinity: odd powers only
            float2 s = v_mul(Bt.v[(ALPHA - 1) * ALPHA + 1], d[1]);
#pragma unroll
            for (int r = 3; r < ALPHA; r += 2) s = v_fma(Bt.v[(ALPHA - 1) * ALPHA + r], d[r], s);
            o[ALPHA - 1] = s;
        }
        // +p / -p pairs: even part E (r = 2, 4, ..), odd part O (r = 1, 3, ..); rows are E + O and E - O
#pragma unroll
        for (int p = 1; p < ALPHA - 1; p += 2) {
            float2 e = v_mul(Bt.v[p * ALPHA + 2], d[2]);
#pragma unroll
            for (int r = 4; r < ALPHA - 1; r += 2) e = v_fma(Bt.v[p * ALPHA + r], d[r], e);
            float2 od = v_mul(Bt.v[p * ALPHA + 1], d[1]);
#pragma unroll
            for (int r = 3; r < ALPHA - 1; r += 2) od = v_fma(Bt.v[p * ALPHA + r], d[r], od);
            o[p] = v_add(e, od);
            o[p + 1] = v_sub(e, od);
        }
    } else {
#pragma unroll
        for (int i = 0; i < ALPHA; ++i) {
            float2 s = v_mul(Bt.v[i * ALPHA], d[0]);
#pragma unroll
            for (int r = 1; r < ALPHA; ++r) s = v_fma(Bt.v[i * ALPHA + r], d[r], s);
            o[i] = s;
        }
    }
}

// ---- stores in the operand formats (lane's channel pair at byte pointers hi / lo) ----
template <int MODE>
__device__ __forceinline__ void put(char* hi, char* lo, float2 v)
{
    if (MODE == STORE_TF32) {
        *reinterpret_cast<float2*>(hi) = make_float2(round_tf32_v(v.x), round_tf32_v(v.y));
    } else if (MODE == STORE_BF16) {
        *reinterpret_cast<__nv_bfloat162*>(hi) = __floats2bfloat162_rn(v.x, v.y);
    } else if (MODE == STORE_TF32_SPLIT) {
        const float2 h = make_float2(round_tf32_v(v.x), round_tf32_v(v.y));
        *reinterpret_cast<float2*>(hi) = h;
        const float2 l = v_sub(v, h);
        *reinterpret_cast<float2*>(lo) = make_float2(round_tf32_v(l.x), round_tf32_v(l.y));
    } else if (MODE == STORE_BF16_SPLIT) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
        const float2 l = v_sub(v, __bfloat1622float2(h));
        *reinterpret_cast<__nv_bfloat162*>(hi) = h;
        *reinterpret_cast<__nv_bfloat162*>(lo) = __floats2bfloat162_rn(l.x, l.y);
    } else {
        *reinterpret_cast<float2*>(hi) = v;
    }
}

// Row pass of one tile: h[r][j'] = sum_j d[r][j] Bt[j'][j].  p0 and p1 (the two channels) point at the 16-byte aligned
// vector of staged row 0 that holds the tile's first column; OFF = that column's index in the vector; row_words = words
// between staged rows.
template <int ALPHA, bool SYM, int OFF>
__device__ __forceinline__ void rows_pass(const float* p0, const float* p1, int row_words, const MatBt2& Bt,
                                          float2 (&h)[ALPHA][ALPHA])
{
    constexpr int NV = (OFF + ALPHA + 3) / 4;
#pragma unroll
    for (int r = 0; r < ALPHA; ++r) {
        float a[4 * NV], b[4 * NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const float4 q = *reinterpret_cast<const float4*>(p0 + r * row_words + 4 * v);
            a[4 * v] = q.x; a[4 * v + 1] = q.y; a[4 * v + 2] = q.z; a[4 * v + 3] = q.w;
            const float4 s = *reinterpret_cast<const float4*>(p1 + r * row_words + 4 * v);
            b[4 * v] = s.x; b[4 * v + 1] = s.y; b[4 * v + 2] = s.z; b[4 * v + 3] = s.w;
        }
        float2 d[ALPHA];
#pragma unroll
        for (int j = 0; j < ALPHA; ++j) d[j] = make_float2(a[OFF + j], b[OFF + j]);
        pass_1d<ALPHA, SYM>(d, h[r], Bt);
    }
}

// Column pass and stores: V[i][j] = sum_r Bt[i][r] h[r][j], transform position xi = i * alpha + j (hi / lo point at
// position (0, 0)).
template <int ALPHA, bool SYM, int MODE>
__device__ __forceinline__ void cols_pass_store(const float2 (&h)[ALPHA][ALPHA], const MatBt2& Bt, char* hi, char* lo,
                                                long long plane_bytes)
{
    const long long row_step = plane_bytes * ALPHA;   // from transform position (i, j) to (i + 1, j)
#pragma unroll
    for (int j = 0; j < ALPHA; ++j) {
        float2 col[ALPHA], o[ALPHA];
#pragma unroll
        for (int r = 0; r < ALPHA; ++r) col[r] = h[r][j];
        pass_1d<ALPHA, SYM>(col, o, Bt);
        char* ph = hi;
        char* pl = lo;
#pragma unroll
        for (int i = 0; i < ALPHA; ++i) {
            put<MODE>(ph, pl, o[i]);
            ph += row_step;
            pl += row_step;
        }
        hi += plane_bytes;
        lo += plane_bytes;
    }
}

// One tile: row pass from the staged rows, column pass, stores; the alpha x alpha intermediate stays in registers.
// `off` = index of the tile's first input column in its 16-byte vector (0..3).
template <int ALPHA, bool SYM>
__device__ __forceinline__ void transform_tile(const float* p0, const float* p1, int row_words, int off, const MatBt2& Bt,
                                               int mode, char* hi, char* lo, long long plane_bytes)
{
    static_assert(ALPHA <= 6, "the intermediate has to fit the registers");
    float2 h[ALPHA][ALPHA];
    switch (off) {
        case 0: rows_pass<ALPHA, SYM, 0>(p0, p1, row_words, Bt, h); break;
        case 1: rows_pass<ALPHA, SYM, 1>(p0, p1, row_words, Bt, h); break;
        case 2: rows_pass<ALPHA, SYM, 2>(p0, p1, row_words, Bt, h); break;
        default: rows_pass<ALPHA, SYM, 3>(p0, p1, row_words, Bt, h); break;
    }
    switch (mode) {
        case STORE_TF32: cols_pass_store<ALPHA, SYM, STORE_TF32>(h, Bt, hi, lo, plane_bytes); break;
        case STORE_BF16: cols_pass_store<ALPHA, SYM, STORE_BF16>(h, Bt, hi, lo, plane_bytes); break;
        case STORE_TF32_SPLIT: cols_pass_store<ALPHA, SYM, STORE_TF32_SPLIT>(h, Bt, hi, lo, plane_bytes); break;
        case STORE_BF16_SPLIT: cols_pass_store<ALPHA, SYM, STORE_BF16_SPLIT>(h, Bt, hi, lo, plane_bytes); break;
        default: cols_pass_store<ALPHA, SYM, STORE_FP32>(h, Bt, hi, lo, plane_bytes); break;
    }
}

// Shared-memory slot of channel c (0..63) of an item: lane l works on channels 2l and 2l + 1 and finds them in slots l
// and 32 + l, so that both reads walk consecutive slots.
__device__ __forceinline__ int slot_of(int c) { return (c & 1) * 32 + (c >> 1); }

template <int ALPHA, bool SYM>
__global__ void __launch_bounds__(kItThreads, 1)
input_transform_ws_kernel(const float* __restrict__ x, const __grid_constant__ CUtensorMap xmap, char* V_hi, char* V_lo,
                          WinoGeom g, InputItems it, int mode, const __grid_constant__ MatBt2 Bt, int* status)
{
    extern __shared__ __align__(128) float s_buf[];
    __shared__ __align__(8) uint64_t full_bar[kItMaxBuffers];
    __shared__ __align__(8) uint64_t empty_bar[kItMaxBuffers];
    __shared__ int4 item_desc[kItMaxBuffers];      // (image, tile row, first tile, channel block) of the item in each buffer
    __shared__ int abort_flag;
    volatile int* abortp = &abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int n_compute = kItWarps - 1;               // warp 0 loads
    const int row_words = kItChannels * it.wb;            // words between staged rows
    if (threadIdx.x == 0) {
        for (int b = 0; b < it.nbuf; ++b) {
            ptx::mbar_init(ptx::smem_u32(&full_bar[b]), 1);
            ptx::mbar_init(ptx::smem_u32(&empty_bar[b]), (uint32_t)n_compute);
        }
        abort_flag = 0;
        ptx::fence_barrier_init();
        ptx::prefetch_tensormap(&xmap);
    }
    __syncthreads();
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();

    // items of this CTA: blockIdx.x, blockIdx.x + gridDim.x, ... (32-bit: the host keeps n_items below 2^31)
    const unsigned first = blockIdx.x, n_items = (unsigned)it.n_items;
    const unsigned n_local = first < n_items ? (n_items - first + gridDim.x - 1) / gridDim.x : 0;
    const int eb = (mode == STORE_BF16 || mode == STORE_BF16_SPLIT) ? 2 : 4;

    if (warp == 0) {
        // ------------------------------- loader -------------------------------
        int b = 0;
        uint32_t round = 0;
        for (unsigned li = 0; li < n_local; ++li) {
            if (round > 0 && !ptx::mbar_wait_relaxed(ptx::smem_u32(&empty_bar[b]), (round - 1) & 1u, abortp)) {
                if (!*abortp && status) atomicCAS(status, 0, kErrInputLoaderWait | (int)(min(li, 0xFFFFu) << 8) | (int)((blockIdx.x & 0x7Fu) << 24));
                *abortp = 1;
                break;
            }
            unsigned item = first + li * gridDim.x;
            const int cb = (int)(item % (unsigned)it.cblocks); item /= (unsigned)it.cblocks;
            const int seg = (int)(item % (unsigned)it.nseg); item /= (unsigned)it.nseg;
            const int ty = (int)(item % (unsigned)g.th);
            const int img = (int)(item / (unsigned)g.th);
            const int tx0 = seg * it.txs;
            const int ih0 = ty * g.m - g.pad, iw0 = tx0 * g.m - g.pad;
            const int a0 = iw0 & ~3;                                     // first staged column, on the vector grid
            const int c0 = cb * kItChannels;
            if (lane == 0) item_desc[b] = make_int4(img, ty, tx0, cb);
            const uint32_t sbuf = ptx::smem_u32(s_buf) + (uint32_t)b * (uint32_t)it.buf_words * 4u;
            const uint32_t bar = ptx::smem_u32(&full_bar[b]);
            if (lane == 0) ptx::mbar_expect_tx(bar, (uint32_t)it.buf_words * 4u);
            __syncwarp();
            // lane = (row, parity): 32 channels of one parity of one input row
            if (lane < 2 * ALPHA) {
                const int r = lane >> 1, par = lane & 1;
                ptx::tma_load_5d(sbuf + (uint32_t)(r * row_words + par * 32 * it.wb) * 4u, &xmap, bar, a0, ih0 + r, par, c0 >> 1, img);
            }
            if (++b == it.nbuf) {
                b = 0;
                ++round;
            }
        }
    } else {
        // ------------------------------- compute -------------------------------
        const int cw = warp - 1;
        const long long plane_bytes = (long long)g.v_plane * eb;
        // Every compute warp waits for every item, in order, and releases it, so that no buffer can run more
        // than one phase ahead of any warp (copies of different items may land out of order, and a parity
        // wait cannot tell a phase that is two behind from one that is done).  Of the item's tiles a
        // warp transforms those whose running index is congruent to it modulo n_compute.
        int b = 0, start = 0;                              // start = (li * it.txs) mod n_compute
        uint32_t round = 0;
        for (unsigned li = 0; li < n_local; ++li) {
            if (!ptx::mbar_wait_relaxed(ptx::smem_u32(&full_bar[b]), round & 1u, abortp)) {
                if (!*abortp && status)
                    atomicCAS(status, 0, kErrInputComputeWait | (int)(min(li, 0xFFFFu) << 8) | (int)((blockIdx.x & 0x7Fu) << 24));
                *abortp = 1;
                break;
            }
            const int4 desc = item_desc[b];
            const int img = desc.x, ty = desc.y, tx0 = desc.z, cb = desc.w;
            const int iw0 = tx0 * g.m - g.pad;
            const int lead = iw0 & 3;                                      // staged columns ahead of the segment
            for (int t = (cw - start + n_compute) % n_compute; t < it.txs; t += n_compute) {
                const int tx = tx0 + t;
                const int c = cb * kItChannels + 2 * lane;
                if (tx < g.tw && c < g.cin_pad) {
                    const long long tile = ((long long)img * g.th + ty) * g.tw + tx;
                    const int s0 = lead + t * g.m;                         // staged column of the tile's first input column
                    const float* p0 = s_buf + (size_t)b * it.buf_words + (size_t)lane * it.wb + (s0 & ~3);
                    const float* p1 = p0 + 32 * it.wb;
                    const long long off = (tile * g.cin_pad + c) * eb;
                    transform_tile<ALPHA, SYM>(p0, p1, row_words, s0 & 3, Bt, mode, V_hi + off, V_lo ? V_lo + off : nullptr,
                                                  plane_bytes);
                }
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&empty_bar[b]));
            start += it.txs % n_compute;
            if (start >= n_compute) start -= n_compute;
            if (++b == it.nbuf) {
                b = 0;
                ++round;
            }
        }
    }
    // After a wait ran out, give copies still in flight time to land before this CTA's shared memory is released.
    if (*abortp) __nanosleep(200000);
}

// Narrow planes whose rows are not 16-byte aligned (14 x 14, 7 x 7, ...), which TMA cannot address row by row: one CTA per
// (image, band of `tr` tile rows, block of 64 channels) copies the band's pixels of the 64 channel planes (at most 256,
// contiguous per channel, so whole warps load although a row is shorter than a warp) into shared memory with plain loads,
// each zero-padded to hp rows x wp columns (image row ih at staged row ih + pad - band * tr * m, image column iw at staged
// column lead + iw; everything else stays zero, which is the convolution's padding and the overhang of the last tiles),
// and then transforms all tiles of the band as the ring kernel does: a tile's vectors are found exactly as there, with wp
// words between staged rows.  hp and wp / 4 are odd, so that 32 lanes reading 128-bit vectors from 32 consecutive planes
// touch every bank once.
//
// A CTA is one trip to memory and one sweep of arithmetic, so its only overlap is with the other CTA of its SM.  Measured,
// transform only: 512 channels 7 x 7 batch 32 5.8 us (two-pass kernel 8.5), 256 channels 14 x 14 batch 32 8.3 us (10.3).
constexpr int kPlaneMaxW = 16;           // (alpha rows of 16 pixels are at most 256)

struct PlaneItems {
    int hp, wp, lead, cblocks, tr, bands;
};

template <int ALPHA, bool SYM>
__global__ void __launch_bounds__(kItThreads, 1)
input_transform_plane_kernel(const float* __restrict__ x, char* V_hi, char* V_lo, WinoGeom g, PlaneItems pi, int mode,
                             const __grid_constant__ MatBt2 Bt)
{
    extern __shared__ __align__(128) float s_buf[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int plane = pi.hp * pi.wp;
    {
        float4* z = reinterpret_cast<float4*>(s_buf);
        for (int i = threadIdx.x; i < kItChannels * plane / 4; i += blockDim.x) z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    ptx::grid_launch_dependents();
    ptx::grid_dependency_wait();
    __syncthreads();
    const int ib = blockIdx.x / pi.cblocks, cb = blockIdx.x - ib * pi.cblocks;
    const int img = ib / pi.bands, band = ib - img * pi.bands;
    const int ty0 = band * pi.tr, tr = min(pi.tr, g.th - ty0);
    const int top = ty0 * g.m - g.pad;                             // image row of staged row 0
    const int ih0 = max(0, top), ih1 = min(g.H, top + (tr - 1) * g.m + ALPHA);
    const int c0 = cb * kItChannels;
    const int n_warps = blockDim.x >> 5, hw = (ih1 - ih0) * g.W;
    {
        // A lane's pixels (lane, lane + 32, ...) land at the same offsets in every plane: decode them once, then
        // copy two channels per step, sixteen loads in flight per lane.  Channels beyond Cin stay zero.
        const size_t plane_hw = (size_t)g.H * g.W;
        const float* xband = x + (size_t)img * g.Cin * plane_hw + (size_t)ih0 * g.W + lane;
        int off[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int p = k * 32 + lane, r = p / g.W;
            off[k] = p < hw ? (ih0 - top + r) * pi.wp + pi.lead + (p - r * g.W) : -1;
        }
        for (int c = warp; c < kItChannels; c += 2 * n_warps) {
            float v[2][8];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int ci = c0 + c + j * n_warps;
                const float* src = xband + (size_t)(ci < g.Cin ? ci : 0) * plane_hw;
#pragma unroll
                for (int k = 0; k < 8; ++k) v[j][k] = (off[k] >= 0 && ci < g.Cin) ? __ldg(src + 32 * k) : 0.0f;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float* dst = s_buf + (size_t)slot_of(c + j * n_warps) * plane;
                if (c0 + c + j * n_warps < g.Cin) {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (off[k] >= 0) dst[off[k]] = v[j][k];
                }
            }
        }
    }
    __syncthreads();
    const int eb = (mode == STORE_BF16 || mode == STORE_BF16_SPLIT) ? 2 : 4;
    const long long plane_bytes = (long long)g.v_plane * eb;
    const int c = c0 + 2 * lane;
    if (c >= g.cin_pad) return;
    for (int ti = warp; ti < tr * g.tw; ti += n_warps) {
        const int ty = ti / g.tw, tx = ti - ty * g.tw;
        const long long tile = ((long long)img * g.th + ty0 + ty) * g.tw + tx;
        const int s0 = pi.lead + tx * g.m - g.pad;                 // staged column of the tile's first input column
        const float* p0 = s_buf + (size_t)lane * plane + (size_t)(ty * g.m) * pi.wp + (s0 & ~3);
        const float* p1 = p0 + (size_t)32 * plane;
        const long long off = (tile * g.cin_pad + c) * eb;
        transform_tile<ALPHA, SYM>(p0, p1, pi.wp, s0 & 3, Bt, mode, V_hi + off, V_lo ? V_lo + off : nullptr, plane_bytes);
    }
}

// Band shape for input_transform_plane_kernel: bands of at most 256 pixels, lower where taller ones would not fill the
// chip.  False for wider planes, and when 64 planes of one tile row do not fit the shared-memory budget.
inline bool plan_plane_items(const WinoGeom& g, int alpha, int num_sms, PlaneItems* pi, size_t* smem)
{
    if (g.W > kPlaneMaxW) return false;
    const int lead = (g.pad + 3) / 4 * 4;
    // columns: the image, and whole 4-wide vectors up to three columns past the last tile
    int wp = lead - g.pad + (g.tw - 1) * g.m + alpha + 3;
    if (wp < lead + g.W) wp = lead + g.W;
    wp = (wp + 3) / 4 * 4;
    if (((wp / 4) & 1) == 0) wp += 4;
    auto rows = [&](int tr) { return ((tr - 1) * g.m + alpha) | 1; };
    auto bytes = [&](int tr) { return (long long)kItChannels * rows(tr) * wp * 4; };
    auto pixels = [&](int tr) { return std::min(g.H, (tr - 1) * g.m + alpha) * g.W; };
    pi->cblocks = (g.cin_pad + kItChannels - 1) / kItChannels;
    const long long per_band = (long long)g.images * pi->cblocks;
    int tr = g.th;
    while (tr > 1 && (bytes(tr) > kItSmemBudget || pixels(tr) > 256 || per_band * ((g.th + tr - 1) / tr) < num_sms)) --tr;
    pi->bands = (g.th + tr - 1) / tr;
    tr = (g.th + pi->bands - 1) / pi->bands;
    if (bytes(tr) > kItSmemBudget || pixels(tr) > 256 || per_band * pi->bands > 2147483647ll) return false;
    pi->tr = tr;
    pi->hp = rows(tr);
    pi->wp = wp;
    pi->lead = lead;
    *smem = (size_t)bytes(tr);
    return true;
}

// True when Bt (alpha x alpha, row-major) has the zero pattern and the +p / -p row symmetry
// that pass_1d<.., SYM = true> assumes.
inline bool bt_has_symmetric_structure(const float* Bt, int alpha)
{
    if (alpha < 4 || (alpha & 1)) return false;
    for (int r = 0; r < alpha; ++r) {
        if ((r & 1) && Bt[r] != 0.0f) return false;                                  // point 0: even powers only
        if (!(r & 1) && Bt[(alpha - 1) * alpha + r] != 0.0f) return false;            // infinity: odd powers only
    }
    for (int p = 1; p < alpha - 1; p += 2) {
        const float* a = Bt + p * alpha;
        const float* b = Bt + (p + 1) * alpha;
        if (a[0] != 0.0f || b[0] != 0.0f || a[alpha - 1] != 0.0f || b[alpha - 1] != 0.0f) return false;
        for (int r = 1; r < alpha - 1; ++r)
            if (b[r] != ((r & 1) ? -a[r] : a[r])) return false;
    }
    return true;
}

// Item geometry.
inline bool plan_input_items(const WinoGeom& g, int alpha, int num_sms, InputItems* it)
{
    it->cblocks = (g.cin_pad + kItChannels - 1) / kItChannels;
    // Candidates: the longest segment for which at least three buffers fit, and up to three finer splits;
    // the one with the shortest schedule wins (rounds of items over the SMs times tiles per item plus one
    // tile's worth of per-item overhead).
    long long best_cost = -1;
    int found = 0;
    for (int nseg = 1; nseg <= g.tw && found < 4; ++nseg) {
        const int txs = (g.tw + nseg - 1) / nseg;
        if (nseg > 1 && txs == (g.tw + nseg - 2) / (nseg - 1)) continue;      // same segment length as before
        const int span = (txs - 1) * g.m + alpha;
        // staged columns: the span, what the vector grid adds in front (up to 3) and what the compute
        // side may read beyond the last tile (whole 4-wide vectors), rounded up to 4 x odd
        int wb = (span + 3 + 3 + 3) / 4 * 4;
        if (((wb / 4) & 1) == 0) wb += 4;
        if (wb > 256) continue;
        const long long bytes = (long long)alpha * kItChannels * wb * 4;
        long long nbuf = kItSmemBudget / bytes;
        if (nbuf < 3 && !(txs == 1 && nbuf >= 2)) continue;
        if (nbuf > kItMaxBuffers) nbuf = kItMaxBuffers;
        const int real_nseg = (g.tw + txs - 1) / txs;
        const long long n_items = (long long)g.images * g.th * real_nseg * it->cblocks;
        if (n_items >= (1ll << 31)) continue;
        const long long rounds = (n_items + num_sms - 1) / num_sms;
        const long long cost = rounds * (txs + 1);
        ++found;
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            it->txs = txs;
            it->nseg = real_nseg;
            it->wb = wb;
            it->nbuf = (int)nbuf;
            it->buf_words = alpha * kItChannels * wb;
            it->n_items = n_items;
        }
    }
    return best_cost >= 0;
}

}  // namespace wino
}  // namespace mnnb
