"""ORACLE — test infrastructure only (tests may import this; the product path never does).

Python-integer restatement of the pre-inference planner (Section 3.2, Eq. 1-5).

The paper selects a computation scheme per convolution layer by minimising a cost
(Eq. 1): an arithmetic count (Eq. 2) that picks the Winograd tile size, the rule that
k = 1 is a matrix product and n-hat = 1 means sliding window (Eq. 3), and a backend term
MUL / FLOPS + t_schedule per operator (Eq. 4, 5).  Read for one GPU whose kernels are
bound by memory traffic, tensor throughput or ALU throughput, the cost of a candidate
scheme is the sum over its kernels of

    max(bytes x c_byte, tensor flops x c_tensor, ALU flops x c_alu) // 10^6 + c_launch

in integer picoseconds; the rate constants are attoseconds per unit, measured once on
the GPU and frozen in a record of sixteen integers (the paper's FLOPS and t_schedule
constants, Appendix C).  The candidate with the smallest cost wins; the first one in
the fixed candidate order wins ties.  Candidates whose predicted error exceeds 0.7 x the
tolerance of the accuracy class are not admissible.  The predicted errors are integers
(parts per million) handed in as a table, so that everything here is a function of
integers: nine layer integers, the options, the sixteen constants and that table.

Candidate order (index into cost_ps): 0 direct; 1 GEMM tf32; 2 GEMM bf16; 3-5 Winograd
m = 2, 4, 6 tf32 x1; 6-8 tf32 x3; 9-11 bf16 x1; 12-14 bf16 x3; 15 Winograd F(2x2,3x3) as one
fused kernel (tf32 x1).

Also here: the paper's own multiplication count (Eq. 2) with the two corrections that make
it comparable across tile sizes (it is a per-tile count; its third term lacks the output
channels), reported beside the choice, and an fp64 restatement of the accuracy model.

Python integers are unbounded; the library saturates every picosecond figure at
2^64 - 2 and so does this file, at the same places.
"""
from __future__ import annotations

from dataclasses import dataclass, field

ALGO_WINOGRAD, ALGO_GEMM, ALGO_DIRECT = 1, 2, 3
OPERAND_TF32, OPERAND_BF16, OPERAND_FP32_REF = 1, 2, 3
PREC_TF32, PREC_BF16 = 0, 1
LHS_PATCHES, LHS_X, LHS_IMPLICIT, LHS_PACKED, LHS_ROWS = 1, 2, 3, 4, 5
INADMISSIBLE = 2 ** 64 - 1
SATURATED = 2 ** 64 - 2
MAX_CHUNK_BYTES = 4 << 30          # V + M of one chunk may not exceed this, whatever the cost says
LHS_X_ERROR_PPM = 340              # truncation of x to TF32 by the tensor core itself (measured)
N_CANDIDATES = 16
FUSED_SLOT = 15


def cdiv(a: int, b: int) -> int:
    return -(-a // b)


def sat(v: int) -> int:
    return min(v, SATURATED)


@dataclass(frozen=True)
class Layer:
    N: int
    Cin: int
    Cout: int
    H: int
    W: int
    k: int
    stride: int = 1
    pad: int = 0
    dil: int = 1
    groups: int = 1

    @property
    def OH(self) -> int:
        return (self.H + 2 * self.pad - self.dil * (self.k - 1) - 1) // self.stride + 1

    @property
    def OW(self) -> int:
        return (self.W + 2 * self.pad - self.dil * (self.k - 1) - 1) // self.stride + 1


@dataclass(frozen=True)
class Options:
    precision: int = PREC_TF32
    operand: int = 0
    passes: int = 0
    force_algo: int = 0
    force_m: int = 0
    points_id: int = 0
    gemm_lhs: int = 0
    fused: int = 0            # 0 planner, 1 never, 2 the fused kernel or nothing


@dataclass
class Choice:
    algo: int = 0
    m: int = 0
    operand: int = 0
    passes: int = 0
    points_id: int = 0
    gemm_lhs: int = 0
    chunk_images: int = 0
    n_chunks: int = 0
    fused: int = 0
    chosen: int = -1
    error_ppm: int = 0
    cost_ps: list = field(default_factory=lambda: [INADMISSIBLE] * N_CANDIDATES)


# ---------------------------------------------------------------------------------------
# One kernel: Eq. 5 with three possible bounds and the launch term.
# ---------------------------------------------------------------------------------------
def kernel_ps(c, mem_as: int = 0, tensor_as: int = 0, alu_as: int = 0) -> int:
    return sat(max(mem_as, tensor_as, alu_as) // 1_000_000 + c[5])


def _bytes_of(operand: int) -> int:
    return 2 if operand == OPERAND_BF16 else 4


def _tensor_rate(c, operand: int) -> int:
    return c[3] if operand == OPERAND_BF16 else c[2]


# ---------------------------------------------------------------------------------------
# Sliding window (Section 3.2 item 3): one kernel, input + output + weights once.
# ---------------------------------------------------------------------------------------
def direct_cost(L: Layer, c) -> int:
    cpg = L.Cin // L.groups
    traffic = 4 * (L.N * L.Cin * L.H * L.W + L.N * L.Cout * L.OH * L.OW + L.Cout * cpg * L.k * L.k)
    flops = 2 * L.N * L.Cout * cpg * L.OH * L.OW * L.k * L.k
    # layers with at most four input channels have a kernel of their own with its own rate,
    # when its transposed weights fit 160 KiB of shared memory
    few_channels = (L.groups == 1 and L.Cin <= 4 and c[9] > 0 and L.N <= 65535
                    and L.Cin * L.k * L.k * (cdiv(L.Cout, 32) * 32) * 4 <= 160 * 1024)
    # c[9] is the rate of the 3 -> Cout, 3x3, stride 2, padding 1 layer on even H and W a multiple of 4 (weights
    # within 48 KiB), which has its own kernel; the other few-channel shapes run at half that rate
    fast = (L.Cin == 3 and L.k == 3 and L.stride == 2 and L.pad == 1 and L.dil == 1 and L.H % 2 == 0 and L.W % 4 == 0
            and 27 * (cdiv(L.Cout, 32) * 32) * 4 <= 48 * 1024)
    if few_channels:
        return kernel_ps(c, mem_as=traffic * c[0], alu_as=flops * (c[9] if fast else 2 * c[9]))
    # c[8] is the rate of layers too small to fill the chip; for k > 1 the lesser of that and 13.3 ns per patch element plus the
    # arithmetic at three tenths of it
    alu = flops * c[8]
    if L.k > 1 and L.Cout > L.groups:                       # (groups of one output channel run a thread per output)
        alu = min(alu, cpg * L.k * L.k * 13300000000 + flops * c[8] * 3 // 10)
    return kernel_ps(c, mem_as=traffic * c[0], alu_as=alu)


# ---------------------------------------------------------------------------------------
# Tiling of the tensor-core contraction: output channels per work item.
# ---------------------------------------------------------------------------------------
def contraction_tiling(tile_blocks: int, positions: int, Cout: int, sms: int):
    """(bn, channel blocks): bn a multiple of 16, at most 256, blocks balanced; among 1x, 2x, 4x the minimum
    number of channel blocks the one with the shortest schedule (rounds over the SMs x operand rows per item)."""
    co16 = cdiv(Cout, 16) * 16
    fewest = cdiv(co16, 256)
    best = None
    for mult in (1, 2, 4):
        bn = cdiv(co16 // 16, fewest * mult) * 16
        if bn < 32 and mult > 1:
            break
        blocks = cdiv(co16, bn)
        length = cdiv(tile_blocks * blocks * positions, sms) * (128 + bn)
        if best is None or length < best[0]:
            best = (length, bn, blocks)
    return best[1], best[2]


def cluster_split(items: int, k_blocks: int, sms: int) -> int:
    """CTAs that share one work item's K loop: doubled while twice as many still fit the SMs and every CTA keeps at least
    four blocks; at most 4, or 8 for up to 8 items."""
    most = 8 if items <= 8 else 4
    n = 1
    while n < most and 2 * n * items <= sms and k_blocks >= 8 * n:
        n *= 2
    return n


def tile_copy_split(items: int, k_blocks: int, sms: int) -> int:
    """The same for the contraction, whose blocks are cheaper: no cut below 36 blocks, 20 where it is by four or eight."""
    n = cluster_split(items, k_blocks, sms)
    return n if k_blocks >= (20 if n > 2 else 36) else 1


# ---------------------------------------------------------------------------------------
# GEMM scheme (k = 1 "is just a matrix multiplication"; k > 1 over gathered patches).
# ---------------------------------------------------------------------------------------
def gemm_may_read_x(L: Layer, operand: int, passes: int) -> bool:
    return (L.k == 1 and L.stride == 1 and L.pad == 0 and L.groups == 1 and operand == OPERAND_TF32
            and passes == 1 and L.H * L.W >= 32 and (L.H * L.W) % 4 == 0)


def packs_lines(L: Layer, operand: int) -> bool:
    """x packed into lines of positions: k in 2..7, stride <= 4, Cin a multiple of 32 or Cin * k <= 32 (BF16: a multiple of
    64), taps reaching at most 600 positions past an output, packed planes of at most 4 GiB."""
    if operand == OPERAND_BF16:
        channels = L.Cin % 64 == 0
    else:
        channels = L.Cin % 32 == 0 or L.Cin * L.k <= 32
    if L.groups != 1 or not 2 <= L.k <= 7 or L.stride > 4 or not channels:
        return False
    reach = (L.k - 1) * L.dil // L.stride
    row, hq = L.OW + reach, L.OH + reach
    strips = cdiv(L.OW, 16)                                # few channels: strips of equal width
    wq = max(row, strips * cdiv(L.OW, strips)) if L.Cin % 32 else row
    cells = L.N * hq * wq
    return (reach * (row + 1) <= 600 and cells < 2 ** 30
            and L.stride ** 2 * (cells + 2048) * (cdiv(L.Cin, 32) * 32) * _bytes_of(operand) <= 4 << 30)


def packed_lines(L: Layer, operand: int, sms: int):
    """Geometry and tiling of the packed-line form, or None: the planes' bytes, the estimated time of the product in ps, whether the
    few-channel form (kernel columns among the elements, rows cut into equal strips of at most 16), the strips' width, and the
    cheapest tiling that fits (output channels bn, mt tiles of 128 cells, g taps per step, stage slots)."""
    bf16, s, offs = operand == OPERAND_BF16, L.stride, {}
    few = L.Cin % (64 if bf16 else 32) != 0
    if few and (bf16 or L.Cin * L.k > 32) or L.k > 7 or s > 4:
        return None
    elems = 32 if few else L.Cin
    k_steps = 3 if few and L.Cin * L.k <= 24 else 4
    for a in range(L.k):
        for b in range(1 if few else L.k):
            offs.setdefault((a * L.dil % s, b * L.dil % s), []).append((a * L.dil // s, b * L.dil // s))
    if len(offs) > 16:
        return None
    qs = [q for group in offs.values() for q in group]

    def pitch(size, out, phases, reach):
        lead = min(cdiv(L.pad - r, s) if r < L.pad else 0 for r in phases)
        end = max((size - 1 + L.pad - r) // s + 1 if size - 1 + L.pad - r >= 0 else 0 for r in phases)
        return max(out, min(out + reach, max(end, out + reach - lead)))

    hq = pitch(L.H, L.OH, [r for r, _ in offs], max(q[0] for q in qs))
    wq = pitch(L.W, L.OW, [r for _, r in offs], max(q[1] for q in qs))
    strips = 1
    if few:
        strips = cdiv(L.OW, 16)
        wq = cdiv(L.OW, strips)
    rows = [[qh * wq + qw for qh, qw in group] for group in offs.values()]
    span, base = max(max(r) - min(r) for r in rows), max(min(r) for r in rows)
    cells, taps = L.N * strips * hq * wq, sum(map(len, rows))
    positions = cells + span + base
    a_bytes = len(rows) * positions * elems * (2 if bf16 else 4)
    if positions >= (1 << 31) - 4096 or a_bytes > 4 << 30:
        return None
    co16, room, best = cdiv(L.Cout, 16) * 16, 207 * 1024, None
    for bn in (256, 128, 64, 32):
        for mt in (1, 2, 4):
            nb = cdiv(co16, bn)
            n = cdiv(cdiv(co16, nb), 16) * 16
            boxes = cdiv(128 * mt + span, 256)
            region = boxes * (cdiv(cdiv(128 * mt + span, boxes), 8) * 8)
            if 2 * mt * n > 512 or (bn > 32 and co16 <= bn // 2) or region > 1024:
                continue
            a_slot, b_tile = region * 128, n * 128
            rounds = cdiv(cdiv(cells, 128 * mt) * nb, sms)
            for g in (3, 2, 1):
                if 2 * a_slot >= room or (room - 2 * a_slot) // (g * b_tile) < (3 if g == 1 else 2):
                    continue
                issue = sum(cdiv(len(r), g) for r in rows) * 194000 + taps * k_steps * 45000
                mma = taps * mt * k_steps * (212 * n + 15000)
                load = (taps * b_tile + len(rows) * a_slot) * 63 // 5
                drain = mt * n * 512 * 28 + 1087000
                item = max(issue, mma, load) * (elems * (2 if bf16 else 4) // 128) + 285000 + mt * 363000
                cost = rounds * max(item, drain) + drain
                if best is None or cost * (100 + 3 * mt) < best[0]:
                    b_slots = min(12, (room - 2 * a_slot) // (g * b_tile))
                    best = (cost * (100 + 3 * mt), cost, dict(bn=n, mt=mt, g=g, b_slots=b_slots,
                                                              a_slots=min(4, (room - b_slots * g * b_tile) // a_slot)))
    return None if best is None else dict(a_bytes=a_bytes, product_ps=best[1], few=few, width=wq, **best[2])


def packed_cost(L: Layer, operand: int, c) -> int:
    """Packed lines: a pass from x to the packed planes at three quarters of the copy rate (half from a stride of four on, in
    TF32), and a product that takes its tiling's estimate or reads the planes and writes y.  TF32: what exceeds two thirds of
    L2, in strips that are not whole sectors, costs five times more; the product's launch hides behind the pack (of few
    channels: 2 us of it)."""
    x, y = 4 * L.N * L.Cin * L.H * L.W, 4 * L.N * L.Cout * L.OH * L.OW
    p = packed_lines(L, operand, c[7] if c[7] > 0 else 148)
    if p is None:
        return INADMISSIBLE
    moved, tf32 = (x + p["a_bytes"]) * c[0] * 4 // 3, operand != OPERAND_BF16
    if tf32 and L.stride >= 4:
        moved = moved * 3 // 2
    kept = c[6] * 2 // 3
    if tf32 and p["few"] and y > kept and (L.OW % 8 or p["width"] % 8):
        y += 5 * (y - kept)
    hidden = 0 if not tf32 else min(2000000, c[5]) if p["few"] else c[5]
    return sat(kernel_ps(c, mem_as=moved) - hidden
               + kernel_ps(c, mem_as=(p["a_bytes"] + y) * c[0], tensor_as=p["product_ps"] * 10 ** 6))


def _mma_cycles(n: int) -> int:
    """An instruction of 128 x n x 32 bytes: 57 cycles for its left operand, more only from 128 channels on."""
    return max(n // 2, 57 + n // 7)


def rows_time(k, m, mode, mt, bn, alpha, taps, rows, b_slot, a_slot, bufs, split, slots, rounds, task_ps=595000):
    """Time of the convolution by rows in ps without its launch."""
    def moved(n):
        return 4096 + 32 * n

    steps, wide = k, 2 if mode == 2 else 1
    tiles = steps * taps * mt
    mma = tiles * (_mma_cycles(2 * bn) + _mma_cycles(bn) if mode == 2 else mode * _mma_cycles(bn)) * 461
    shared = tiles * (moved(2 * bn) + moved(bn) if mode == 2 else mode * moved(bn)) + steps * b_slot + a_slot
    x_bytes, tasks = rows * 64 * (1 if m == 1 else alpha), cdiv(rows, 32) * (1 if m == 1 else 2)
    serial = cdiv(tasks, 10) * task_ps if m == 1 else cdiv(tasks, 12) * 1418000
    stage = max(mma, (shared * 2 + x_bytes * (12 if m == 1 else 3)) * 193 // 100, serial) + steps * 51500
    drain, loop = 1098000 + 5700 * mt * bn * alpha * wide, slots * stage + 672000
    cost = rounds * max(loop, drain) + drain if bufs == 2 else rounds * (loop + drain)
    return cost + (2348000 + 4000 * mt * bn * m if split > 1 else 0) - 446000


def rows_tiling(L: Layer, m: int, passes: int, sms: int):
    """The one-kernel convolution by rows: m outputs of a row per cell (one-dimensional Winograd F(2, 3); 1: the definition), kernel
    rows as shifts.  The cheapest tiling that fits as a dict with its time in ps, or None."""
    k = L.k
    if not (m == 2 and k == 3 or m == 1 and k in (2, 3, 5, 7)):
        return None
    alpha = 1 if m == 1 else m + k - 1
    taps = k if m == 1 else alpha

    def pitch(size, out, reach):
        return max(out, min(out + reach, max(size + L.pad, out + reach - L.pad)))

    hq = pitch(L.H, L.OH, k - 1)
    wq = pitch(L.W, L.OW, k - 1) if m == 1 else cdiv(L.OW, m)
    cells, span = L.N * hq * wq, (k - 1) * wq + (k - 1 if m == 1 else 0)
    if cells >= (1 << 31) - 65536 or span > 2048:
        return None
    stages, co16, room, best = cdiv(L.Cin, 16), cdiv(L.Cout, 16) * 16, 213 * 1024, None
    from_memory = m == 1 and 4 * L.N * (L.Cin * L.H * L.W + L.Cout * L.OH * L.OW) > 16000000
    for mode in ([1] if passes == 1 else [3] if m == 2 else [2, 3]):
        halves, wide = (1 if mode == 1 else 2), (2 if mode == 2 else 1)
        for mt in ((1, 2) if m == 1 else (1,)):
            seen = set()
            for nb in range(1, co16 // 16 + 1):
                bn = cdiv(cdiv(co16, nb), 16) * 16
                if bn in seen:
                    continue
                seen.add(bn)
                if wide * bn > 256 or alpha * mt * wide * bn > 512:
                    continue
                bufs = 2 if 2 * alpha * mt * wide * bn <= 512 else 1
                if mt == 2 and bufs == 1 or m == 1 and mode == 3 and k == 7 and mt == 1:
                    continue
                rows = cdiv(128 * mt + span, 8) * 8
                a_slot, b_slot = alpha * halves * rows * 32, taps * halves * bn * 32
                if 2 * a_slot + 3 * b_slot > room:
                    continue
                items = cdiv(cells, 128 * mt) * nb
                if items >= 1 << 31:
                    continue
                for split in (1, 2, 4, 8):
                    if split > 1 and (mt > 1 or m == 1 and mode == 3 and k >= 5 or items * split > sms or split == 4 and items > 32 or split == 8 and items > 8
                                      or 2 * stages < 3 * split or bn * m * 512 > room):
                        break
                    args = (k, m, mode, mt, bn, alpha, taps, rows, b_slot, a_slot, bufs, split, cdiv(stages, split), cdiv(items * split, sms))
                    cost = rows_time(*args)
                    if best is None or cost < best["time_ps"]:
                        best = dict(time_ps=cost, memory_ps=rows_time(*args, 900000) if from_memory else cost, mode=mode, mt=mt, bn=bn, split=split, items=items, rows=rows)
    return best


# Row-wise Winograd, hi + lo BF16: F(4, 3), F(4, 5), F(2, 7); parts per million as measured, rounded up.
ROW_WISE_PPM = {3: 20, 5: 30, 7: 30}


def row_wise_tiling(L: Layer, m: int, sms: int):
    """Three kernels that transform along the rows only: bytes of V and M and the cheapest tiling of the product, or None."""
    k, alpha, reach = L.k, m + L.k - 1, L.k - 1
    hq = max(L.OH, min(L.OH + reach, max(L.H + L.pad, L.OH + reach - L.pad)))
    tiles_w = cdiv(L.OW, m)
    T, cin_pad = L.N * hq * tiles_w, cdiv(L.Cin, 8) * 8
    v, mm = 4 * alpha * T * cin_pad, 4 * alpha * L.Cout * (cdiv(T, 32) * 32)
    if T >= (1 << 31) - 65536 or v + mm > 4 << 30:
        return None
    co16, room, best = cdiv(L.Cout, 16) * 16, 207 * 1024, None
    for mt in (1, 2):
        for nb in range(cdiv(co16, 256), min(64, co16 // 16) + 1):
            bn = cdiv(cdiv(co16, nb), 16) * 16
            need = 128 * mt + reach * tiles_w
            boxes = cdiv(need, 256)
            rows = boxes * (cdiv(cdiv(need, boxes), 8) * 8)
            a_slot, b_slot = 2 * rows * 64, 2 * bn * 64
            items = cdiv(T, 128 * mt) * nb * alpha
            if 2 * mt * bn > 512 or 2 * a_slot + 3 * b_slot > room or items >= 1 << 31:
                continue
            mma = 6 * mt * k * max(bn // 2, 57 + bn // 7) * 555
            load = (a_slot + k * b_slot) * 63 // 5
            drain = mt * bn * 512 * 28 + 1087000
            cost = cdiv(items, sms) * max(cdiv(cin_pad, 32) * max(mma, load) + 285000, drain) + drain
            if best is None or cost < best["product_ps"]:
                best = dict(product_ps=cost, v=v, m=mm, bn=bn, mt=mt)
    return best


def row_wise_cost(L: Layer, t, c) -> int:
    x, y = 4 * L.N * L.Cin * L.H * L.W, 4 * L.N * L.Cout * L.OH * L.OW
    return sat(kernel_ps(c, mem_as=(x + t["v"]) * c[0] * 3 // 2) + kernel_ps(c, mem_as=(t["m"] + y) * c[0] * 3 // 2) + t["product_ps"] + c[5])


def gemm_cost(L: Layer, operand: int, lhs, c) -> int:
    """lhs: LHS_PATCHES (gather kernel + GEMM), LHS_X / True (the GEMM reads x itself), LHS_IMPLICIT (the patches are
    gathered by producer warps inside the GEMM kernel)."""
    lhs_x = lhs is True or lhs == LHS_X
    implicit = lhs is not True and lhs == LHS_IMPLICIT
    b = _bytes_of(operand)
    Kp = cdiv(L.Cin * L.k * L.k, 8) * 8
    T = L.N * L.OH * L.OW
    x_bytes = 4 * L.N * L.Cin * L.H * L.W
    y_bytes = 4 * L.N * L.Cout * L.OH * L.OW
    v_bytes = T * Kp * b
    u_bytes = L.Cout * Kp * b
    sms = c[7] if c[7] > 0 else 148
    # the contraction as it is scheduled: rounds of work items, each a serial loop over 128-byte blocks of K
    # paced by the tensor core or by the delivery of the operand tiles (16 ps per byte), the accumulator drained
    # (45 ps per byte, half a microsecond of hand-over) while the next item's loop runs; one drain is exposed
    tile_blocks = L.N * cdiv(cdiv(L.H * L.W, 32), 4) if lhs_x else cdiv(T, 128)
    bn, co_blocks = contraction_tiling(tile_blocks, 1, L.Cout, sms)
    rounds = cdiv(tile_blocks * co_blocks, sms)
    k_elems = 128 // b
    k_blocks = cdiv(Kp, k_elems)
    deliver_ps = (128 * 128 + bn * 128) * 16
    mma_ps = sat(2 * 128 * bn * k_elems * _tensor_rate(c, operand) * sms // 1_000_000)
    drain_ps = 128 * bn * 4 * 45
    if implicit:
        # only the weight tile is delivered; the gather of 128 x 32 patch elements (c[13] attoseconds each) paces a block too
        # (c[13] is measured on the tap-major gather, Cin a multiple of 32; other channel counts gather element-wise, about 2x)
        block_ps = max(bn * 128 * 16, mma_ps, sat(128 * 32 * c[13] * (1 if L.Cin % 32 == 0 else 2) // 1_000_000))
        item_i = max(k_blocks * block_ps, drain_ps + 500_000)
        return kernel_ps(c, mem_as=(x_bytes + u_bytes + y_bytes) * c[0], tensor_as=(rounds * item_i + drain_ps) * 1_000_000)
    item_ps = max(k_blocks * max(deliver_ps, mma_ps), drain_ps + 500_000)
    serial_as = (rounds * item_ps + drain_ps) * 1_000_000
    if lhs_x:
        return kernel_ps(c, mem_as=(x_bytes + u_bytes + y_bytes) * c[0], tensor_as=serial_as)
    # the patch gather at its measured rate relative to a plain copy: 1.5x (1x1 stride-1: a transposition),
    # 3x (k > 1, staged through shared memory), 5x (strided 1x1, element-wise)
    transposition = L.k == 1 and L.stride == 1 and L.pad == 0 and (L.H * L.W) % 4 == 0
    twice_factor = 3 if transposition else (6 if L.k > 1 else 10)
    gather = kernel_ps(c, mem_as=(x_bytes + v_bytes) * c[0] * twice_factor // 2)
    contract = kernel_ps(c, mem_as=(v_bytes + u_bytes + y_bytes) * c[0], tensor_as=serial_as)
    return sat(gather + contract)


def staged_gather(L: Layer):
    """(time in ps of a CTA's serial loads, CTAs) of the gather staged through shared memory, or (0, 0) where it does not
    serve: output positions in segments of at most 64 columns, at most 64 positions per CTA (128 / 256 for short rows of V), a
    slab of at most 64 groups of four patch elements whose input region fits 9216 floats; half a microsecond per step of
    region rows (eight warps), 0.2 us for each further 32 columns."""
    if L.k == 1:
        return 0, 0
    groups, k2 = cdiv(L.Cin * L.k * L.k, 8) * 2, L.k * L.k
    width = cdiv(L.OW, cdiv(L.OW, 64))
    rows = max(1, min((256 if groups <= 16 else 128 if groups <= 32 else 64) // width, L.OH))
    rh = (rows - 1) * L.stride + (L.k - 1) * L.dil + 1
    rw = (width - 1) * L.stride + (L.k - 1) * L.dil + 1

    def channels(q):
        return (4 * q + k2 - 2) // k2 + 1
    fitting = [q for q in {min(q, groups) for q in range(8, 65, 8)} if channels(q) * rh * rw <= 9216]
    if not fitting:
        return 0, 0
    slab, lanes = max(fitting), 32
    while lanes > 1 and lanes // 2 >= rw:
        lanes //= 2
    return (cdiv(channels(slab) * rh, 8 * (32 // lanes)) * (300000 + 200000 * cdiv(rw, lanes)),
            L.N * cdiv(L.OH, rows) * cdiv(L.OW, width) * cdiv(groups, slab))


def patch_operand_time(L: Layer, lhs, c):
    """Time in ps of the TF32 GEMM scheme over patches that are written first (LHS_PATCHES) or gathered by producer warps
    (LHS_IMPLICIT), the K loop cut over clusters; chooses between the two where the loop is cut."""
    sms = c[7] if c[7] > 0 else 148
    Kp, T = cdiv(L.Cin * L.k * L.k, 8) * 8, L.N * L.OH * L.OW
    bn, co_blocks = contraction_tiling(cdiv(T, 128), 1, L.Cout, sms)
    items = cdiv(T, 128) * co_blocks
    rounds, split = cdiv(items, sms), (cluster_split if lhs == LHS_IMPLICIT else tile_copy_split)(items, cdiv(Kp, 32), sms)
    x, y, v, u = 4 * L.N * L.Cin * L.H * L.W, 4 * L.N * L.Cout * L.OH * L.OW, T * Kp * 4, L.Cout * Kp * 4
    drain = 128 * bn * 4 * 45
    if lhs == LHS_IMPLICIT:
        gather = min(1024000, 128 * 32 * c[13] // 10 ** 6)  # ps per block of 128 x 32 elements, measured
        block = max(gather * 15 // 8 if L.Cin % 32 else gather * 2 if L.stride >= 4 else gather, bn * 128 * 16)
        fixed, traffic = 0, x + u + y
    else:
        serial, ctas = staged_gather(L)
        moved = (x + v) * c[0] // 10 ** 6
        if serial:
            fixed = 2500000 + max(serial, serial * cdiv(ctas, 4 * sms) * 3 // 4) + moved * 6 // 5
        else:
            fixed = max(2500000, moved * 5)
        block = max((128 * 128 + bn * 128) * 16, 2 * 128 * bn * 32 * c[2] * sms // 10 ** 6) * 3 // 5
        traffic = v + u + y
    item = max(cdiv(cdiv(Kp, 32), split) * block, 128 * bn * 4 * 82 + 1250000 if lhs == LHS_IMPLICIT and split == 1 else drain + 500000)
    fixed += 3000000 if split > 1 else 0                    # what a cut costs
    return fixed + kernel_ps(c, mem_as=traffic * c[0], tensor_as=(rounds * item + (drain // 2 if split > 1 else drain)) * 10 ** 6)


# ---------------------------------------------------------------------------------------
# Winograd F(m x m, k x k) as three kernels (Eq. 6), chunked over the batch.
# ---------------------------------------------------------------------------------------
def winograd_supported(m: int, k: int) -> bool:
    return m in (2, 4, 6) and k in (2, 3, 5, 7) and m + k - 1 <= 12


def winograd_cost(L: Layer, m: int, operand: int, passes: int, c):
    """(chunk_images, n_chunks, cost_ps)."""
    alpha = m + L.k - 1
    a2 = alpha * alpha
    tiles_img = cdiv(L.OH, m) * cdiv(L.OW, m)
    Cp = cdiv(L.Cin, 8) * 8
    b_el = _bytes_of(operand) * (2 if passes == 3 else 1)
    per_image = a2 * tiles_img * Cp * b_el + a2 * L.Cout * tiles_img * 4
    fits_l2 = c[6] // per_image
    cap = max(1, MAX_CHUNK_BYTES // per_image)
    chunk = L.N if L.N < cap else cdiv(L.N, cdiv(L.N, cap))
    n_chunks = cdiv(L.N, chunk)
    # one chunk: input transform, contraction, output transform
    n = chunk
    v = n * a2 * tiles_img * Cp * b_el
    mm = n * a2 * L.Cout * tiles_img * 4
    u = a2 * L.Cout * Cp * b_el
    x = 4 * n * L.Cin * L.H * L.W
    y = 4 * n * L.Cout * L.OH * L.OW
    c_vm = c[1] if fits_l2 >= chunk else c[0]
    # ALU work of the transforms: 2 alpha^3 multiply-adds per (tile, channel) on the input side (the first term
    # of Eq. 2), m alpha (alpha + m) on the output side (its third term); from alpha = 8 a lane holds one channel
    # instead of a pair and sweeps over the tile's columns: x2 at alpha = 8, x2.25 at alpha = 10, x4 at alpha = 12
    # (in quarters: 8, 9, 16 against 4)
    quarters = 16 if alpha >= 12 else (9 if alpha >= 10 else (8 if alpha >= 8 else 4))
    t_in = kernel_ps(c, mem_as=x * c[0] + v * c_vm, alu_as=quarters * alpha * a2 * n * tiles_img * L.Cin * c[4])
    # the contraction's work items (128 tiles x bn channels x one position) go over the SMs in rounds, and the
    # tensor time is that of full rounds
    sms = c[7] if c[7] > 0 else 148
    tile_blocks = cdiv(n * tiles_img, 128)
    _, co_blocks = contraction_tiling(tile_blocks, a2, L.Cout, sms)
    items = tile_blocks * co_blocks * a2
    tensor = 2 * a2 * L.Cout * Cp * n * tiles_img * passes * _tensor_rate(c, operand) // items * (cdiv(items, sms) * sms)
    t_con = kernel_ps(c, mem_as=(v + mm) * c_vm + u * c[0], tensor_as=tensor)
    t_out = kernel_ps(c, mem_as=mm * c_vm + y * c[0], alu_as=2 * m * alpha * (alpha + m) * n * tiles_img * L.Cout * c[4])
    return chunk, n_chunks, sat(n_chunks * sat(t_in + t_con + t_out))


# ---------------------------------------------------------------------------------------
# Winograd F(2x2, 3x3) as ONE kernel: transforms in the producer and epilogue warps, the sixteen
# accumulators of a block of 128 output channels x 32 tiles in tensor memory.  HBM sees x, y and U only.
# ---------------------------------------------------------------------------------------
def fused_supported(L: Layer) -> bool:
    return L.k == 3 and L.stride == 1 and L.dil == 1 and L.groups == 1 and L.pad <= 2


def fused_cost(L: Layer, c) -> int:
    tiles = L.N * cdiv(L.OH, 2) * cdiv(L.OW, 2)
    sms = c[7] if c[7] > 0 else 148
    x = 4 * L.N * L.Cin * L.H * L.W
    y = 4 * L.N * L.Cout * L.OH * L.OW
    u = 16 * L.Cout * L.Cin * 4
    co_blocks = cdiv(L.Cout, 128)
    items = cdiv(tiles, 32) * co_blocks
    rounds = cdiv(items, sms)
    k_blocks = cdiv(L.Cin, 32)
    # an item is a serial loop over blocks of 32 input channels; a block costs the delivery of sixteen
    # 128 x 32 weight tiles from L2 to the SM (c[10] attoseconds per byte and SM) or sixty-four small MMAs
    # whose pace the shared-memory reads of the 128-row operand set (c[11] picoseconds per block), whichever
    # is larger; then the epilogue (c[12] picoseconds per item) before the next item's MMAs may start
    block_ps = max(16 * 128 * 32 * 4 * c[10] // 1_000_000, c[11])
    item_ps = k_blocks * block_ps + c[12]
    serial_as = rounds * item_ps * 1_000_000
    # x comes from HBM once; the other channel blocks find it in L2
    return kernel_ps(c, mem_as=(x + y + u) * c[0] + (co_blocks - 1) * x * c[1], tensor_as=serial_as)


# ---------------------------------------------------------------------------------------
# The selection (Eq. 1, Eq. 3).
# ---------------------------------------------------------------------------------------
def _candidates():
    out = [(ALGO_DIRECT, 0, 0, 0), (ALGO_GEMM, 0, OPERAND_TF32, 1), (ALGO_GEMM, 0, OPERAND_BF16, 1)]
    for operand, passes in ((OPERAND_TF32, 1), (OPERAND_TF32, 3), (OPERAND_BF16, 1), (OPERAND_BF16, 3)):
        for m in (2, 4, 6):
            out.append((ALGO_WINOGRAD, m, operand, passes))
    out.append((ALGO_WINOGRAD, 2, OPERAND_TF32, 1))       # slot 15: the fused kernel
    return out


def best_points(ppm, m, k, operand, passes):
    """(points_id, ppm) with the lowest predicted error; the first wins ties.  ``ppm`` maps
    (m, k, points_id, operand, passes) to parts per million, missing or negative = not available."""
    best = (0, -1)
    for pid in (1, 2, 3):
        p = ppm.get((m, k, pid, operand, passes), -1)
        if p < 0:
            continue
        if best[0] == 0 or p < best[1]:
            best = (pid, p)
    return best


def plan(L: Layer, o: Options, c, ppm) -> Choice:
    """The planner's decision for the list-driven case (no off-list forced combination)."""
    ch = Choice()
    gate = (10000 if o.precision == PREC_BF16 else 1000) * 7 // 10
    fully_forced = o.force_m != 0 and o.operand != 0 and o.passes != 0
    wino_shape = L.stride == 1 and L.dil == 1 and L.groups == 1 and 2 <= L.k <= 7
    side = {}
    for i, (algo, m, operand, passes) in enumerate(_candidates()):
        if o.fused == 2 and i != FUSED_SLOT:
            continue
        if o.force_algo != 0 and o.force_algo != algo:
            continue
        if algo == ALGO_DIRECT:
            if o.operand in (0, OPERAND_FP32_REF) or o.force_algo == ALGO_DIRECT:
                ch.cost_ps[i] = direct_cost(L, c)
            continue
        if o.operand != 0 and o.operand != operand:
            continue
        if o.passes != 0 and o.passes != passes:
            continue
        if algo == ALGO_GEMM:
            if L.groups != 1 or o.force_m != 0:
                continue
            p = ppm.get((1, L.k, 0, operand, passes), -1)
            if p < 0:
                continue
            if p > gate and not (o.operand != 0 and o.force_algo == ALGO_GEMM):
                continue
            x_ok = gemm_may_read_x(L, operand, passes)
            implicit_ok = operand == OPERAND_TF32 and passes == 1
            if o.gemm_lhs == LHS_X and not x_ok:
                continue
            if o.gemm_lhs == LHS_IMPLICIT and not implicit_ok:
                continue
            costs = {LHS_PATCHES: gemm_cost(L, operand, LHS_PATCHES, c)}
            if x_ok:
                costs[LHS_X] = gemm_cost(L, operand, LHS_X, c)
            if implicit_ok:
                costs[LHS_IMPLICIT] = gemm_cost(L, operand, LHS_IMPLICIT, c)
            # left operand: as asked for, else the cheapest that applies (patch matrix, x itself, implicit gather;
            # earlier in this order on ties; the implicit gather only once its rate constant is known)
            lhs = o.gemm_lhs
            if lhs == 0:
                lhs = LHS_PATCHES
                if x_ok and costs[LHS_X] < costs[lhs]:
                    lhs = LHS_X
                # (plain pointwise layers keep the tuned paths: measured, the implicit gather never beat them there)
                if implicit_ok and not (L.k == 1 and L.stride == 1) and c[13] > 0 and costs[LHS_IMPLICIT] < costs[lhs]:
                    lhs = LHS_IMPLICIT
                costs_of = lhs
                # items so few that their K loop is cut over clusters: the implicit gather instead of patches where that takes
                # less; else packed lines where they apply.  Booked at the cost of the operand chosen above.
                sms = c[7] if c[7] > 0 else 148
                blocks = cdiv(L.N * L.OH * L.OW, 128)
                _, co_blocks = contraction_tiling(blocks, 1, L.Cout, sms)
                cut = cluster_split(blocks * co_blocks, cdiv(cdiv(L.Cin * L.k * L.k, 8) * 8, 32), sms) > 1
                if implicit_ok and cut and not (L.k == 1 and L.stride == 1) and c[13] > 0:
                    if lhs == LHS_PATCHES and patch_operand_time(L, LHS_IMPLICIT, c) < patch_operand_time(L, LHS_PATCHES, c):
                        lhs = LHS_IMPLICIT
                elif packs_lines(L, operand):
                    # TF32: unless estimated at 6/5 of the other operand's time or more
                    tf32 = implicit_ok and lhs != LHS_X
                    if packed_cost(L, operand, c) * (5 if tf32 else 1) < (6 * patch_operand_time(L, lhs, c) if tf32 else costs[lhs]):
                        lhs = LHS_PACKED
                costs[lhs] = costs[costs_of]
            if lhs == LHS_X:
                p = max(p, LHS_X_ERROR_PPM)
            side[i] = dict(lhs=lhs, ppm=p)
            ch.cost_ps[i] = costs[lhs]
            continue
        # Winograd
        fused = i == FUSED_SLOT
        if fused and (o.fused == 1 or not fused_supported(L) or c[10] <= 0 or c[11] <= 0):
            continue
        if not wino_shape or not winograd_supported(m, L.k):
            continue
        if o.force_m != 0 and o.force_m != m:
            continue
        if o.points_id == 0:
            pid, p = best_points(ppm, m, L.k, operand, passes)
        else:
            pid, p = o.points_id, ppm.get((m, L.k, o.points_id, operand, passes), -1)
        if pid == 0 or p < 0:
            continue
        if p > gate and not fully_forced:
            continue
        if fused:
            side[i] = dict(pid=pid, ppm=p, chunk=L.N, n_chunks=1)
            ch.cost_ps[i] = fused_cost(L, c)
        else:
            chunk, n_chunks, cost = winograd_cost(L, m, operand, passes, c)
            side[i] = dict(pid=pid, ppm=p, chunk=chunk, n_chunks=n_chunks)
            ch.cost_ps[i] = cost
    best = -1
    for i in range(N_CANDIDATES):
        if ch.cost_ps[i] != INADMISSIBLE and (best < 0 or ch.cost_ps[i] < ch.cost_ps[best]):
            best = i
    # BF16 class: packed lines in BF16 take over from a scheme that is neither faster nor expected to be more accurate
    if best not in (-1, 2) and side.get(2, {}).get("lhs") == LHS_PACKED and side[2]["ppm"] <= side.get(best, {}).get("ppm", 0):
        cost = packed_cost(L, OPERAND_BF16, c)
        if cost < ch.cost_ps[best]:
            ch.cost_ps[2], best = cost, 2
    # The convolution by rows takes over where nothing is forced, it is estimated faster than a tensor-core scheme (by what is held
    # against it: the estimates' measured errors) and not expected to be less accurate: as candidate 2 (the definition) or 12 (Winograd m = 2).
    held = 10 if L.W % 4 and L.k <= 5 else 15 if L.k == 7 and best >= 3 and _candidates()[best][1] == 6 else 11
    rows, row_wise, ppm_before = False, False, side.get(best, {}).get("ppm", 0)
    winograd_before = best >= 3              # only then another Winograd form
    free = o.force_algo == o.force_m == o.operand == o.passes == o.points_id == o.gemm_lhs == o.fused == 0
    if free and wino_shape and best > 0:
        for m in (1, 2):
            passes, slot = (1 if o.precision == PREC_BF16 else 3), (2 if m == 1 else 12)
            t = None if m == 2 and (passes == 1 or not winograd_before) else rows_tiling(L, m, passes, c[7] if c[7] > 0 else 148)
            if t is None:
                continue
            pid, p = (0, ppm.get((1, L.k, 0, OPERAND_BF16, passes), -1)) if m == 1 else best_points(ppm, m, L.k, OPERAND_BF16, passes)
            now = ch.cost_ps[best]
            lines = not rows and side[best].get("lhs") == LHS_PACKED
            cost = t["time_ps"] + c[5]
            if lines:                           # by their own time; BF16: x from memory, and two overlapping kernels
                now, cost = min(now, packed_cost(L, _candidates()[best][2], c)), (t["memory_ps"] if passes == 1 else t["time_ps"]) + c[5]
            faster = (cost < now if rows else cost * 9 < now * 10 if lines and passes == 3 else cost * 19 + 80000000 < now * 20 if lines else cost * held < now * 10)
            if p < 0 or p > ppm_before or not faster:
                continue
            best, rows, ch.cost_ps[slot] = slot, True, cost
            side[slot] = dict(lhs=LHS_ROWS, ppm=p, pid=pid, chunk=L.N, n_chunks=1)
        if winograd_before and o.precision == PREC_TF32 and L.k in ROW_WISE_PPM and ROW_WISE_PPM[L.k] <= ppm_before:
            m = 2 if L.k == 7 else 4
            t = row_wise_tiling(L, m, c[7] if c[7] > 0 else 148)
            if t is not None and row_wise_cost(L, t, c) * (10 if rows else held) < ch.cost_ps[best] * 10:
                best, rows, row_wise = (12 if m == 2 else 13), False, True
                ch.cost_ps[best] = row_wise_cost(L, t, c)
                side[best] = dict(ppm=ROW_WISE_PPM[L.k], pid=best_points(ppm, m, L.k, OPERAND_BF16, 3)[0], chunk=L.N, n_chunks=1)
    if best < 0:
        return ch
    algo, m, operand, passes = _candidates()[best]
    ch.chosen, ch.algo, ch.operand, ch.passes = best, algo, operand, 3 if rows and o.precision == PREC_TF32 else passes
    ch.error_ppm = side.get(best, {}).get("ppm", 0)
    if algo == ALGO_WINOGRAD:
        ch.m, ch.points_id = m, side[best]["pid"]
        ch.chunk_images, ch.n_chunks = side[best]["chunk"], side[best]["n_chunks"]
        ch.fused = 1 if best == FUSED_SLOT else 2 if rows else 3 if row_wise else 0
    else:
        ch.m, ch.points_id, ch.chunk_images, ch.n_chunks = 1, 0, L.N, 1
        ch.gemm_lhs = side[best]["lhs"] if algo == ALGO_GEMM else 0
    return ch


# ---------------------------------------------------------------------------------------
# The paper's own count (Eq. 2), made comparable across n: it is a per-tile count, so it is multiplied by
# the number of tiles, and its third term (the output transform) gets the o_c factor it lacks as printed.
# ---------------------------------------------------------------------------------------
def paper_multiplications(L: Layer, n: int) -> int:
    a = n + L.k - 1
    tiles = L.N * cdiv(L.OH, n) * cdiv(L.OW, n)
    return tiles * (2 * L.Cin * a ** 3 + L.Cin * L.Cout * a ** 2 + L.Cout * n * a * (2 * n + L.k - 1))


def paper_choice(L: Layer, sizes=(1, 2, 4, 6)):
    """(n-hat, [count per n]): Eq. 2's argmin over the tile sizes; n-hat = 1 means sliding window (Eq. 3)."""
    counts = [paper_multiplications(L, n) for n in sizes]
    return sizes[counts.index(min(counts))], counts


# ---------------------------------------------------------------------------------------
# Accuracy model: F(m, k) on a fixed pseudo-random problem in fp64 with U and V rounded to the operand
# format (optionally split into hi + lo), relative L2 error against the plain correlation, in ppm.
# Same data recipe as the library's gate (a 64-bit LCG, sums of twelve uniforms), restated with NumPy.
# ---------------------------------------------------------------------------------------
def _lcg_normalish(seed: int, count: int):
    import numpy as np
    s = seed
    out = np.empty(count, dtype=np.float64)
    mask = (1 << 64) - 1
    for i in range(count):
        acc = 0.0
        for _ in range(12):
            s = (s * 6364136223846793005 + 1442695040888963407) & mask
            acc += (s >> 11) * (1.0 / 9007199254740992.0)
        out[i] = acc - 6.0
    return out


def _round_bits(a, bits):
    """fp32(a) rounded to `bits` explicit mantissa bits, ties to even, as fp64."""
    import numpy as np
    f = np.asarray(a, dtype=np.float64).astype(np.float32)
    u = f.view(np.uint32).astype(np.uint64)
    drop = 23 - bits
    if drop > 0:
        lsb = (u >> np.uint64(drop)) & np.uint64(1)
        u = u + np.uint64((1 << (drop - 1)) - 1) + lsb
        u = u & ~np.uint64((1 << drop) - 1)
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def accuracy_ppm(m: int, k: int, points_id: int, operand: int, passes: int, generate=None) -> int:
    """``generate(m, k, points_id)`` returns (A, G, Bt) as exact rationals (the oracle's generator)."""
    import math

    import numpy as np
    bits = {OPERAND_TF32: 10, OPERAND_BF16: 7, OPERAND_FP32_REF: 23}[operand]
    C, CO, TILES = 64, 4, 16
    alpha = m + k - 1
    a2 = alpha * alpha
    seed = 0x9E3779B97F4A7C15 ^ (m * 1000 + k * 10)
    draws = _lcg_normalish(seed, CO * C * k * k + TILES * C * a2)
    w = (draws[:CO * C * k * k] * (1.0 / math.sqrt(C * k * k))).astype(np.float32).astype(np.float64).reshape(CO, C, k, k)
    x = draws[CO * C * k * k:].astype(np.float32).astype(np.float64).reshape(TILES, C, alpha, alpha)

    def split(v):
        hi = _round_bits(v, bits)
        lo = _round_bits(v.astype(np.float32).astype(np.float64) - hi, bits) if passes == 3 else np.zeros_like(hi)
        return hi, lo

    if m == 1 and points_id == 0:
        wk = w.reshape(CO, C * k * k)              # alpha = k here: a tile is one k x k patch
        xk = x.reshape(TILES, C * k * k)
        wh, wl = split(wk)
        xh, xl = split(xk)
        ref = xk @ wk.T
        got = xh @ wh.T + xh @ wl.T + xl @ wh.T
    else:
        A, G, Bt = generate(m, k, points_id)
        A = np.array([[float(v) for v in r] for r in A])
        G = np.array([[float(v) for v in r] for r in G])
        Bt = np.array([[float(v) for v in r] for r in Bt])
        U = np.einsum("ia,ocab,jb->ocij", G, w, G)
        V = np.einsum("ia,tcab,jb->tcij", Bt, x, Bt)
        Uh, Ul = split(U)
        Vh, Vl = split(V)
        M = (np.einsum("ocij,tcij->toij", Uh, Vh) + np.einsum("ocij,tcij->toij", Ul, Vh)
             + np.einsum("ocij,tcij->toij", Uh, Vl))
        M = M.astype(np.float32).astype(np.float64)
        got = np.einsum("ia,toij,jb->toab", A, M, A)
        ref = np.zeros((TILES, CO, m, m))
        for i in range(k):
            for j in range(k):
                ref += np.einsum("oc,tcab->toab", w[:, :, i, j], x[:, :, i:i + m, j:j + m])
    rel = math.sqrt(float(((got - ref) ** 2).sum()) / float((ref ** 2).sum()))
    return int(math.ceil(rel * 1e6))


# ---------------------------------------------------------------------------------------
# Strassen's stopping rule (Eq. 9) for [n x k] x [k x m]: recurse while the multiplications saved outnumber
# the additions added, both counted alike.
# ---------------------------------------------------------------------------------------
def strassen_rule(m: int, n: int, k: int) -> bool:
    if min(m, n, k) < 2:
        return False
    mh, nh, kh = m // 2, n // 2, k // 2
    return m * n * k - 7 * mh * nh * kh > 4 * mh * kh + 4 * nh * kh + 7 * mh * nh
