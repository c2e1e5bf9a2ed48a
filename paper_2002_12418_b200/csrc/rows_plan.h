// Geometry and tiling of the one-kernel convolution by rows (rows_conv.cu).  Host only, integers only.
//
// One axis of the kernel (the "line") is handled by one-dimensional Winograd F(m, k) or, with m = 1, by the definition; the other
// axis by shifting the operand.  The work is laid out in cells: a cell (n, i, j) is a tile of m outputs along the line, cells are
// numbered over N x Hq x Wq, and kernel row a of a cell reads the transformed input a * Wq cells further on.  Rows and images
// share their zero padding as in the packed lines (line_plan.h).
#pragma once
#include <cstdint>

namespace mnnb {

constexpr int kRowsChannels = 16;        // input channels per stage: one tensor-core step of BF16
constexpr int kRowsMaxA = 4, kRowsMaxB = 10;
constexpr int kRowsSmemBytes = 214 * 1024;
constexpr int kRowsMaxAlpha = 4;

struct RowsShape {
    int N, Cin, Cout, H, W, kh, kw, pad_h, pad_w, OH, OW;
    int m;                               // outputs per cell along the width (1: kw shifted taps instead of a transform)
    int passes;                          // 1: BF16 operands, 3: hi + lo
};

struct RowsPlan {
    RowsShape s;
    int alpha;                           // operand planes: m + kw - 1, or 1 where m = 1
    int steps, taps;                     // a stage: steps (kernel rows) of taps weight tiles: kh of alpha, or of kw where m = 1; k x 1: one of k
    int step_rows, tap_rows;             // cells between consecutive steps, and between taps where m = 1
    int n_acc;                           // accumulators per tile of 128 cells
    int Hq, Wq;
    long long T;                         // cells
    int mode;                            // 1: one product; 3: three; 2: three as two instructions (rows_conv.cu)
    int mt, rows, rows_pad;              // tiles of 128 cells per item; staged rows per plane (multiples of 8 and 32)
    int k_slots;                         // stages of 16 input channels
    int bn, n_co_blocks, split, a_slots, b_slots, acc_bufs;
    long long n_tile_blocks, n_items, u_bytes;
    long long time_ps;                   // estimated time of the kernel without its launch
    long long memory_ps;                 // the same where x has to come from memory
};

bool rows_plan(const RowsShape& s, int num_sms, RowsPlan* p);

}  // namespace mnnb
