// Geometry and tiling of the packed-line convolution (line_conv.cu).  Host only, integers only.
//
// x is re-laid ("packed") into planes of positions, a position being one 128-byte row per block of 32 TF32 or 64 BF16 operand elements:
//     A [plane][position][elements]           elements = input channels, a multiple of 32 (TF32) or 64 (BF16)
// A position is a cell (n, i, j) of a grid of N x Hq x Wq cells, a cell an output position, a plane one of the input phases
// of the stride.  Kernel tap (a, b) reads, for every cell, the cell `shift` positions further on in its phase's plane, so a
// tap is a change of the operand's start row and nothing is gathered.  Rows and images share their zero padding: the cells
// right of a row are the left padding of the next one.
// Layers with few channels (Cin * k <= 32) put the k columns of a kernel row into the elements too, (ci, b) -> ci * k + b;
// then planes are the row phases, a tap is a kernel row, and no cell needs its neighbours along the row: the image is cut
// into strips of about 16 columns, N x strips x Hq x Wq cells, so that a kernel row is a shift of 16 positions and not of a
// whole row (3 -> 64 7x7 stride 2 at 224 x 224, batch 32: a region of 304 instead of 592 positions per 256 cells).
#pragma once
#include <algorithm>
#include <cstdint>

namespace mnnb {

constexpr int kLineMaxTaps = 49, kLineMaxPlanes = 16, kLineMaxA = 4, kLineMaxB = 12;
constexpr int kLineSmemBytes = 208 * 1024;
constexpr int kLineMaxRegion = 1024;     // positions staged at a time

// Cells of one axis: `out` outputs, `lead` zero cells in front, data cells end before `end`, taps reach `reach` cells past an
// output.  The smallest pitch that lets the zero cells behind the data be the next line's leading ones.
inline int axis_pitch(int out, int lead, int end, int reach)
{
    return std::max(out, std::min(out + reach, std::max(end, out + reach - lead)));
}

struct LineShape {
    int N, Cin, Cout, H, W, k, stride, dil, pad, OH, OW;
    int bf16;                            // operand elements: BF16 (not in the few-channel form), else TF32
};

struct LinePlan {
    LineShape s;
    int few;                             // the few-channel form
    int elems, blocks;                   // elements per position, in blocks of 128 bytes
    int k_steps;                         // tensor-core steps of 32 bytes in a block (3 for few channels of at most 24 elements, else 4)
    int n_planes, phase_h[kLineMaxPlanes], phase_w[kLineMaxPlanes];
    int strips, Hq, Wq;                  // strips: 1 unless few
    long long T, P;                      // cells; positions per plane in memory
    int n_taps, n_groups;
    int tap_id[kLineMaxTaps];            // in the order of the weight tiles: a * k + b, or a (few)
    int tap_rel[kLineMaxTaps];           // first row inside the staged region
    int group_plane[kLineMaxPlanes], group_base[kLineMaxPlanes], group_first[kLineMaxPlanes], group_taps[kLineMaxPlanes];
    // tiling
    int bn, n_co_blocks, mt;             // output channels, blocks of them, and tiles of 128 cells per work item
    int region, boxes, box_rows;         // staged positions = boxes * box_rows
    int taps_per_step;                   // weight tiles that share a slot and a barrier
    int a_slots, b_slots;
    long long n_tile_blocks, n_items, a_bytes, u_bytes;
    long long loop_ps;                   // estimated time of the product without its launch and fill
};

// Fills *p; false where the form does not apply (channels not a multiple of 32 and not few, region or phases too large).
bool line_plan(const LineShape& s, int num_sms, LinePlan* p);

}  // namespace mnnb
