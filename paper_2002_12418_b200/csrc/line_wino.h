// Row-wise Winograd (line_wino.cu): one-dimensional F(m, k) along the rows, kernel rows as shifts of the staged operand.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "kernels.h"

namespace mnnb {

struct LineWinoShape {
    int N, Cin, Cout, H, W, k, pad, OH, OW, m;
};

// Lines are the rows of the padded images, neighbours sharing their zero rows: Hq per image; a line has `tiles_w` tiles of m
// outputs, T = N * Hq * tiles_w.  Tap (kernel row) a of a tile reads V[xi] a * tiles_w tiles further on.
struct LineWinoPlan {
    LineWinoShape s;
    int alpha, Hq, tiles_w, cin_pad, blocks;     // blocks of 32 channels
    long long T;
    int mt, bn, n_co_blocks, rows, boxes, box_rows, a_slots, b_slots, tmem_cols;
    long long n_tile_blocks, n_items, m_row_stride, u_bytes, v_bytes, m_bytes;     // u, v: hi and lo halves together
    long long product_ps;                        // estimated time of the product without its launch
};

struct LineWino {
    LineWinoPlan p;
    CUtensorMap map_v_hi, map_v_lo, map_u_hi, map_u_lo;
    int num_sms = 0;
    bool ready = false;
};

bool line_wino_plan(const LineWinoShape& s, int num_sms, LineWinoPlan* p);
cudaError_t line_wino_setup(LineWino* lw, void* V, void* U, const char** why);
// U [xi][kernel row][Cout][cin_pad], hi then lo, from w and the one-dimensional matrix G [alpha][k].
cudaError_t launch_line_wino_weights(const LineWinoPlan& p, const float* w, void* U, const float* G, cudaStream_t stream);
// M[xi][co][t] = sum over kernel rows and channels of V[xi][t + a * tiles_w][ci] * U[xi][a][co][ci].
cudaError_t launch_line_wino_product(const LineWino& lw, float* M, int* status, cudaStream_t stream);

}  // namespace mnnb
