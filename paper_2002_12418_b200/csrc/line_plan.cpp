// Geometry and tiling of the packed-line convolution.
#include "line_plan.h"

#include <algorithm>
#include <cstring>

namespace mnnb {

namespace {

long long cdiv(long long a, long long b) { return (a + b - 1) / b; }
long long rup(long long a, long long b) { return cdiv(a, b) * b; }

}  // namespace

bool line_plan(const LineShape& s, int num_sms, LinePlan* p)
{
    std::memset(p, 0, sizeof(*p));
    p->s = s;
    const int block = s.bf16 ? 64 : 32, eb = s.bf16 ? 2 : 4;
    p->few = s.Cin % block != 0;
    if (p->few && (s.bf16 || s.Cin * s.k > 32)) return false;
    if (s.k > 7 || s.stride > 4) return false;
    p->elems = p->few ? 32 : s.Cin;
    p->blocks = p->elems / block;
    p->k_steps = p->few && s.Cin * s.k <= 24 ? 3 : 4;

    // phases and taps, grouped by phase
    struct Tap { int id, qh, qw; };
    Tap taps[kLineMaxPlanes][kLineMaxTaps];
    int n_in[kLineMaxPlanes] = {0};
    int qh_max = 0, qw_max = 0;
    const int kb = p->few ? 1 : s.k;
    for (int a = 0; a < s.k; ++a)
        for (int b = 0; b < kb; ++b) {
            const int rh = a * s.dil % s.stride, rw = b * s.dil % s.stride;
            int ph = 0;
            while (ph < p->n_planes && !(p->phase_h[ph] == rh && p->phase_w[ph] == rw)) ++ph;
            if (ph == p->n_planes) {
                if (ph == kLineMaxPlanes) return false;
                p->phase_h[ph] = rh;
                p->phase_w[ph] = rw;
                ++p->n_planes;
            }
            taps[ph][n_in[ph]++] = {p->few ? a : a * s.k + b, a * s.dil / s.stride, b * s.dil / s.stride};
            qh_max = std::max(qh_max, a * s.dil / s.stride);
            qw_max = std::max(qw_max, b * s.dil / s.stride);
        }
    for (int ax = 0; ax < 2; ++ax) {
        const int in = ax ? s.W : s.H, out = ax ? s.OW : s.OH, reach = ax ? qw_max : qh_max;
        int lead = 1 << 30, end = 0;
        for (int i = 0; i < p->n_planes; ++i) {
            const int r = ax ? p->phase_w[i] : p->phase_h[i];
            lead = std::min(lead, r < s.pad ? (int)cdiv(s.pad - r, s.stride) : 0);
            end = std::max(end, in - 1 + s.pad - r >= 0 ? (in - 1 + s.pad - r) / s.stride + 1 : 0);
        }
        const int pitch = axis_pitch(out, lead, end, reach);
        if (ax) p->Wq = pitch;
        else p->Hq = pitch;
    }
    p->strips = 1;
    if (p->few) {
        p->strips = (int)cdiv(s.OW, 16);
        p->Wq = (int)cdiv(s.OW, p->strips);
    }
    int span = 0, max_base = 0;
    p->n_groups = p->n_planes;
    for (int g = 0; g < p->n_planes; ++g) {
        p->group_plane[g] = g;
        p->group_first[g] = p->n_taps;
        p->group_taps[g] = n_in[g];
        int lo = 1 << 30;
        for (int t = 0; t < n_in[g]; ++t) lo = std::min(lo, taps[g][t].qh * p->Wq + taps[g][t].qw);
        p->group_base[g] = lo;
        max_base = std::max(max_base, lo);
        for (int t = 0; t < n_in[g]; ++t) {
            const int rel = taps[g][t].qh * p->Wq + taps[g][t].qw - lo;
            p->tap_id[p->n_taps] = taps[g][t].id;
            p->tap_rel[p->n_taps++] = rel;
            span = std::max(span, rel);
        }
    }
    p->T = (long long)s.N * p->strips * p->Hq * p->Wq;
    p->P = p->T + span + max_base;       // rows past the end of a plane read as zeros or as the next plane, for no valid cell
    if (p->P >= (1ll << 31) - 4096) return false;
    p->a_bytes = (long long)p->n_planes * p->P * p->elems * eb;
    p->u_bytes = (long long)p->n_taps * s.Cout * p->elems * eb;
    if (p->a_bytes > (4ll << 30)) return false;

    // Tiling: the shortest loop, rounds of items over the SMs times the pace of a block of 128 bytes: an issuing thread's
    // serial time (0.2 us per step and 45 ns per instruction; each tile of cells has a thread of its own), the tensor core's
    // (15 ns + 0.21 ns per output channel and instruction) or the delivery of regions and weight tiles (12.6 ps per byte and
    // SM), whichever is longest; then what an item costs besides or its drain.  Fitted to 690 measured
    // products (20 layers, every tiling) to 8 %; the choice is within 5 % of the best of most, 11 % at worst, with 3 % held
    // against each further tile of an item.
    // Two tiles of 128 channels rather than one of 256: half the weight bytes and two issuing threads (256 channels 28 x 28
    // dilation 2 batch 16 34.3 -> 31.5 us, 64 channels 56 x 56 batch 64 59 -> 39).
    const int co16 = (int)rup(s.Cout, 16);
    long long best = -1;
    for (int bn = 256; bn >= 32; bn /= 2)
        for (int mt = 1; mt <= 4; mt *= 2) {
            const int nb = (int)cdiv(co16, bn), b_n = (int)rup(cdiv(co16, nb), 16);
            if (2 * mt * b_n > 512 || (bn > 32 && co16 <= bn / 2)) continue;
            const int rows = 128 * mt + span, boxes = (int)cdiv(rows, 256), box_rows = (int)rup(cdiv(rows, boxes), 8);
            if (boxes * box_rows > kLineMaxRegion) continue;
            const long long a_slot = (long long)boxes * box_rows * 128, b_tile = (long long)b_n * 128;
            const long long tile_blocks = cdiv(p->T, 128 * mt), items = tile_blocks * nb;
            if (items >= (1ll << 31)) continue;
            const long long rounds = cdiv(items, num_sms);
            for (int g = 3; g >= 1; --g) {
                const long long room = kLineSmemBytes - 1024;
                int b_slots = (int)((room - 2 * a_slot) / (g * b_tile));
                if (2 * a_slot >= room || b_slots < (g == 1 ? 3 : 2)) continue;
                b_slots = std::min(b_slots, kLineMaxB);
                const int a_slots = (int)std::min<long long>(kLineMaxA, (room - b_slots * g * b_tile) / a_slot);
                long long steps = 0;
                for (int i = 0; i < p->n_groups; ++i) steps += cdiv(p->group_taps[i], g);
                const long long issue = steps * 194000 + (long long)p->n_taps * p->k_steps * 45000;
                const long long mma = (long long)p->n_taps * mt * p->k_steps * (212 * b_n + 15000);
                const long long load = (p->n_taps * b_tile + p->n_groups * a_slot) * 63 / 5;
                const long long drain = (long long)mt * b_n * 128 * 4 * 28 + 1087000;
                const long long cost = rounds * std::max(std::max(issue, std::max(mma, load)) * p->blocks + 285000 + mt * 363000, drain) + drain;
                if (best < 0 || cost * (100 + 3 * mt) < best) {
                    best = cost * (100 + 3 * mt);
                    p->bn = b_n;
                    p->n_co_blocks = nb;
                    p->mt = mt;
                    p->region = boxes * box_rows;
                    p->boxes = boxes;
                    p->box_rows = box_rows;
                    p->taps_per_step = g;
                    p->a_slots = a_slots;
                    p->b_slots = b_slots;
                    p->n_tile_blocks = tile_blocks;
                    p->n_items = items;
                    p->loop_ps = cost;
                }
            }
        }
    return best >= 0;
}

}  // namespace mnnb
