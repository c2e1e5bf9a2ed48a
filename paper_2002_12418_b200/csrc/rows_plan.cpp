// Geometry and tiling of the one-kernel convolution by rows.
#include "rows_plan.h"

#include <algorithm>
#include <cstring>

#include "line_plan.h"

namespace mnnb {

namespace {

long long cdiv(long long a, long long b) { return (a + b - 1) / b; }
long long rup(long long a, long long b) { return cdiv(a, b) * b; }

}  // namespace

bool rows_plan(const RowsShape& s, int num_sms, RowsPlan* p)
{
    std::memset(p, 0, sizeof(*p));
    p->s = s;
    const int line = s.kw == 1 ? s.kh : s.kw;                  // the axis whose taps share a step
    if (!((s.m == 2 && s.kw == 3) || (s.m == 1 && (line == 2 || line == 3 || line == 5 || line == 7))) || s.kh > 7) return false;
    p->alpha = s.m == 1 ? 1 : s.m + s.kw - 1;
    p->n_acc = p->alpha;
    p->Hq = axis_pitch(s.OH, s.pad_h, s.H + s.pad_h, s.kh - 1);
    p->Wq = s.m == 1 ? axis_pitch(s.OW, s.pad_w, s.W + s.pad_w, s.kw - 1) : (int)cdiv(s.OW, s.m);
    p->T = (long long)s.N * p->Hq * p->Wq;
    const bool column = s.m == 1 && s.kw == 1;                 // k x 1: the taps go down the column, all in one step
    p->steps = column ? 1 : s.kh;
    p->taps = column ? s.kh : s.m == 1 ? s.kw : p->alpha;
    p->step_rows = p->Wq;
    p->tap_rows = column ? p->Wq : 1;
    const int span = (s.kh - 1) * p->Wq + (s.m == 1 ? s.kw - 1 : 0);
    if (p->T >= (1ll << 31) - 65536 || span > 2048) return false;
    p->k_slots = (int)cdiv(s.Cin, kRowsChannels);
    const int co16 = (int)rup(s.Cout, 16);
    // A round of producer tasks: 0.6 us where x comes from the L2, 0.9 from memory.  176 BF16 layers whose x and y together pass 16 MB, each
    // with other inputs than the call before: the estimate is 9 % off (rms) with the second, 18 % with the first; 72 smaller ones 21 and 12 %.
    const bool from_memory = s.m == 1 && 4ll * s.N * ((long long)s.Cin * s.H * s.W + (long long)s.Cout * s.OH * s.OW) > 16000000;
    long long best = -1;
    for (int mode = s.passes == 1 ? 1 : s.m == 2 ? 3 : 2; mode <= s.passes; ++mode)
      for (int mt = 1; mt <= (s.m == 1 ? 2 : 1); ++mt)
        for (int nb = 1; nb <= (int)cdiv(co16, 16); ++nb) {
            const int bn = (int)rup(cdiv(co16, nb), 16);
            const int hl = mode == 1 ? 1 : 2, wide = mode == 2 ? 2 : 1;
            if (wide * bn > 256 || p->n_acc * mt * wide * bn > 512) continue;
            if (nb > 1 && (int)rup(cdiv(co16, nb - 1), 16) == bn) continue;
            const int bufs = 2 * p->n_acc * mt * wide * bn <= 512 ? 2 : 1;
            if (s.m == 1 && mode == 3 && line == 7 && mt == 1) continue;      // (never the shortest of 60000 layers, clusters with three products from k = 5 on in two of them: not compiled)
            if (mt == 2 && bufs == 1) continue;      // (256 channels 56 x 56 batch 64, one product: 310 us, one tile 218)
            const int rows = (int)rup(128 * mt + span, 8);
            const long long a_slot = (long long)p->alpha * hl * rows * 32, b_slot = (long long)p->taps * hl * bn * 32;
            const long long room = kRowsSmemBytes - 1024;
            if (2 * a_slot + 3 * b_slot > room) continue;
            const int b_slots = (int)std::min<long long>(kRowsMaxB, (room - 2 * a_slot) / b_slot);
            const int a_slots = (int)std::min<long long>(kRowsMaxA, (room - b_slots * b_slot) / a_slot);
            const long long tile_blocks = cdiv(p->T, 128 * mt), items = tile_blocks * nb;
            if (items >= (1ll << 31)) continue;
            for (int split = 1; split <= 8; split *= 2) {
                // (clusters of four and eight that do not all fit the GPCs at once run in two waves: 36 of four 10 -> 20 us)
                // A CTA may have one stage beside others with two: 112 channels (seven stages) 10 x 10 one image in four 7.5 us, in two 10.3 (three
                // Winograd kernels 7.1 to 8), 96 channels 5 x 7 four images 7.5 and 9.5 (7.5 to 8).
                if (split > 1 && (mt > 1 || (s.m == 1 && mode == 3 && line >= 5) || items * split > num_sms || (split == 4 && items > 32) || (split == 8 && items > 8) || 2 * p->k_slots < 3 * split ||
                                  (long long)bn * s.m * 512 > room))
                    break;
                // A stage: the instructions of its weight tiles (57 cycles for the left operand, more only from 128 channels on), or what
                // they and the producers move through shared memory and the L1, or the producers' serial time; and the waits of its
                // steps.  Fitted to 797 measured tilings of 135 layers: 4 % off in the median, 13 % at
                // the ninth decile.
                auto cycles = [](long long n) { return std::max(n / 2, 57 + n / 7); };
                auto bytes = [](long long n) { return 4096 + 32 * n; };
                const long long rounds = cdiv(items * split, num_sms), slots = cdiv(p->k_slots, split), tiles = (long long)p->steps * p->taps * mt;
                const long long mma = tiles * (mode == 2 ? cycles(2 * bn) + cycles(bn) : mode * cycles(bn)) * 461;
                const long long moved = tiles * (mode == 2 ? bytes(2 * bn) + bytes(bn) : mode * bytes(bn)) + p->steps * b_slot + a_slot;
                const long long x_bytes = (long long)rows * 64 * (s.m == 1 ? 1 : p->alpha), tasks = cdiv(rows, 32) * (s.m == 1 ? 1 : 2);
                const long long drain = 1098000 + 5700ll * mt * bn * p->n_acc * wide;
                auto time = [&](long long task_ps) {
                    const long long serial = s.m == 1 ? cdiv(tasks, 10) * task_ps : cdiv(tasks, 12) * 1418000;
                    const long long stage = std::max(std::max(mma, (moved * 2 + x_bytes * (s.m == 1 ? 12 : 3)) * 193 / 100), serial) + p->steps * 51500ll;
                    const long long loop = slots * stage + 672000;
                    return (bufs == 2 ? rounds * std::max(loop, drain) + drain : rounds * (loop + drain)) +
                           (split > 1 ? 2348000 + 4000ll * mt * bn * s.m : 0) - 446000;
                };
                const long long cost = time(595000);
                if (best < 0 || cost < best) {
                    best = cost;
                    p->mt = mt;
                    p->mode = mode;
                    p->rows = rows;
                    p->rows_pad = (int)rup(rows, 32);
                    p->bn = bn;
                    p->n_co_blocks = nb;
                    p->split = split;
                    p->a_slots = a_slots;
                    p->b_slots = b_slots;
                    p->acc_bufs = bufs;
                    p->n_tile_blocks = tile_blocks;
                    p->n_items = items;
                    p->time_ps = cost;
                    p->memory_ps = from_memory ? time(900000) : cost;
                }
            }
        }
    if (best < 0) return false;
    p->u_bytes = (long long)p->n_co_blocks * p->k_slots * p->steps * p->taps * (p->mode == 1 ? 1 : 2) * p->bn * 32;
    return true;
}

}  // namespace mnnb
