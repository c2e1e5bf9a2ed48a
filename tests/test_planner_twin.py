"""The planner (Section 3.2, Eq. 1-5) against its Python-integer twin, and the twin against what
arithmetic fixes.  No GPU: planning is host work.

* every layer of configs 0-4, both batch sizes, both accuracy classes, two calibration records
  (built-in and a perturbed one): every cost_ps[i] and every field of the decision bit-equal;
* two fresh processes given the same frozen record return byte-identical mnn_conv_info;
* the accuracy gate's integers (ppm) reproduced by an fp64 restatement of the model on the exact
  rational generator's matrices;
* the twin itself: hand-computed costs, the tie-break, saturation, Eq. 2 on a worked example.
"""
import functools
import json
import os
import subprocess
import sys

import pytest

from oracle import planner_twin as T
from oracle import winograd_exact as wx
from paper_2002_12418_b200 import binding as B
from paper_2002_12418_b200 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@functools.lru_cache(maxsize=None)
def ppm_table():
    """The accuracy model's integers, read through the ABI, as the twin's input table."""
    t = {}
    for k in (1, 2, 3, 5, 7):
        for operand in (B.OPERAND_TF32, B.OPERAND_BF16):
            for passes in (1, 3):
                t[(1, k, 0, operand, passes)] = B.mnn_accuracy_ppm(1, k, 0, operand, passes)
                if k == 1:
                    continue
                for m in (2, 4, 6):
                    if m + k - 1 > 12:
                        continue
                    for pid in (1, 2, 3):
                        try:
                            t[(m, k, pid, operand, passes)] = B.mnn_accuracy_ppm(m, k, pid, operand, passes)
                        except B.MnnError:
                            pass
    return t


def all_layers():
    out = []
    for cfg in (W.config0(), W.config1(1), W.config1(32), W.config2(1), W.config2(32), W.config3(1), W.config3(64),
                W.config4(64)):
        out += cfg
    return out


def twin_layer(l):
    return T.Layer(l.N, l.Cin, l.Cout, l.H, l.W, l.k, l.stride, l.pad, l.dilation, l.groups)


def compare(l, opts_kw, twin_kw, cal):
    o = B.make_opts(groups=l.groups, relu=l.relu, **opts_kw)
    plan = B.mnn_conv_plan_ex(l.N, l.Cin, l.Cout, l.H, l.W, l.k, l.stride, l.pad, l.dilation, o)
    info = B.mnn_conv_plan_query(plan)
    B.mnn_conv_destroy(plan)
    ch = T.plan(twin_layer(l), T.Options(**twin_kw), cal, ppm_table())
    what = "%s %s" % (l.name, opts_kw)
    assert list(info.cost_ps) == ch.cost_ps, what
    got = (info.chosen_candidate, info.algo, info.m, info.operand, info.passes, info.points_id, info.gemm_lhs,
           info.chunk_images, info.n_chunks, info.fused, info.predicted_error_ppm)
    want = (ch.chosen, ch.algo, ch.m, ch.operand, ch.passes, ch.points_id, ch.gemm_lhs, ch.chunk_images, ch.n_chunks,
            ch.fused, ch.error_ppm)
    assert got == want, what
    n_hat, counts = T.paper_choice(twin_layer(l))
    assert (info.paper_n_hat, list(info.paper_mul)) == (n_hat, counts), what
    return info


@pytest.fixture()
def restore_calibration():
    B.lib()
    before = B.mnn_get_calibration()
    yield before
    B.mnn_set_calibration(before)


PERTURBED = [211000, 61000, 2500, 900, 35000, 5100000, 40 << 20, 132, 480000, 45000, 15000, 900000, 2500000, 90000000, 0, 0]


@pytest.mark.parametrize("record", ["builtin", "perturbed"])
def test_every_config_layer_matches_the_twin(restore_calibration, record):
    cal = list(restore_calibration) if record == "builtin" else PERTURBED
    B.mnn_set_calibration(cal)
    assert B.mnn_get_calibration() == cal
    n = 0
    for l in all_layers():
        for prec in (B.PREC_TF32, B.PREC_BF16):
            compare(l, dict(precision=prec), dict(precision=prec), cal)
            n += 1
    assert n >= 200


def test_forced_options_match_the_twin(restore_calibration):
    cal = list(restore_calibration)
    l = W.config1(32)[1]
    cases = [
        (dict(force_algo=B.ALGO_WINOGRAD), dict(force_algo=T.ALGO_WINOGRAD)),
        (dict(force_algo=B.ALGO_GEMM), dict(force_algo=T.ALGO_GEMM)),
        (dict(force_algo=B.ALGO_DIRECT), dict(force_algo=T.ALGO_DIRECT)),
        (dict(force_m=4), dict(force_m=4)),
        (dict(operand=B.OPERAND_BF16), dict(operand=T.OPERAND_BF16)),
        (dict(passes=3), dict(passes=3)),
        (dict(points_id=1), dict(points_id=1)),
        (dict(fused=B.FUSED_NEVER), dict(fused=1)),
        (dict(fused=B.FUSED_ONLY), dict(fused=2)),
        (dict(force_m=6, operand=B.OPERAND_TF32, passes=1), dict(force_m=6, operand=T.OPERAND_TF32, passes=1)),
    ]
    for okw, tkw in cases:
        compare(l, okw, tkw, cal)
    pw = W.config3(64)[2]
    for lhs in (B.GEMM_LHS_PATCHES, B.GEMM_LHS_X, B.GEMM_LHS_IMPLICIT):
        compare(pw, dict(gemm_lhs=lhs), dict(gemm_lhs=lhs), cal)
    s2 = W.config2(32)[5]                                   # 3x3 stride 2: patches or the implicit gather
    for lhs in (B.GEMM_LHS_PATCHES, B.GEMM_LHS_IMPLICIT):
        compare(s2, dict(force_algo=B.ALGO_GEMM, gemm_lhs=lhs), dict(force_algo=T.ALGO_GEMM, gemm_lhs=lhs), cal)
    fast = list(cal)
    fast[13] = 1000                                         # a gather that costs nothing: the planner takes it by itself
    B.mnn_set_calibration(fast)
    info = compare(s2, dict(force_algo=B.ALGO_GEMM), dict(force_algo=T.ALGO_GEMM), fast)
    assert info.gemm_lhs == B.GEMM_LHS_IMPLICIT


def test_fused_candidate_disappears_without_its_constants(restore_calibration):
    cal = list(restore_calibration)
    cal[10] = 0
    B.mnn_set_calibration(cal)
    info = compare(W.config1(32)[0], {}, {}, cal)
    assert info.cost_ps[15] == B.COST_INADMISSIBLE


def test_very_large_layers_saturate_instead_of_wrapping(restore_calibration):
    cal = list(restore_calibration)
    # just under the 2^40-element limit of the ABI: attosecond products pass 2^64
    big = W.ConvLayer("huge", 4096, 1024, 1024, 500, 500, 3, 1, 1, seed=1)
    info = compare(big, {}, {}, cal)
    finite = [c for c in info.cost_ps if c != B.COST_INADMISSIBLE]
    small = W.ConvLayer("small", 1, 1024, 1024, 500, 500, 3, 1, 1, seed=1)
    info_small = compare(small, {}, {}, cal)
    for a, b in zip(info.cost_ps, info_small.cost_ps):
        if a != B.COST_INADMISSIBLE:
            assert a > b                                   # 4096 images never cost less than one
    assert finite


def test_two_fresh_processes_return_identical_bytes():
    code = r"""
import ctypes, sys, json
sys.path.insert(0, %r)
from paper_2002_12418_b200 import binding as B
from paper_2002_12418_b200 import workloads as W
B.mnn_set_calibration(%r)
out = []
for cfg in (W.config1(32), W.config3(64), W.config4(64)):
    for l in cfg:
        for prec in (0, 1):
            p = B.mnn_conv_plan_ex(l.N, l.Cin, l.Cout, l.H, l.W, l.k, l.stride, l.pad, l.dilation,
                                   B.make_opts(groups=l.groups, relu=l.relu, precision=prec))
            out.append(bytes(B.mnn_conv_plan_query(p)).hex())
            B.mnn_conv_destroy(p)
print(json.dumps(out))
""" % (ROOT, PERTURBED)
    runs = [subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, check=True).stdout for _ in range(2)]
    a, b = json.loads(runs[0]), json.loads(runs[1])
    assert len(a) == 2 * (4 + 27 + 4) and a == b


# ---------------------------------------------------------------------------
# The accuracy gate's integers.
# ---------------------------------------------------------------------------
@pytest.mark.parametrize("m,k", [(1, 1), (1, 3), (1, 7), (2, 3), (4, 3), (6, 3), (2, 5), (4, 5), (2, 7), (4, 7), (6, 7)])
def test_accuracy_model_matches_its_fp64_restatement(m, k):
    B.lib()
    for operand in (B.OPERAND_TF32, B.OPERAND_BF16):
        for passes in (1, 3):
            for pid in ((0,) if m == 1 else (1, 2, 3)):
                try:
                    lib = B.mnn_accuracy_ppm(m, k, pid, operand, passes)
                except B.MnnError:
                    continue
                twin = T.accuracy_ppm(m, k, pid, operand, passes, generate=wx.generate)
                # the two sum in different orders: equal up to the last unit of a value that is rounded up
                assert abs(lib - twin) <= max(1, lib // 10 ** 9), (m, k, pid, operand, passes, lib, twin)


def test_accuracy_gate_separates_what_the_tolerances_separate():
    t = ppm_table()
    # one TF32 pass meets 1e-3 (with the 0.7 margin) only at m = 2; three passes always do for alpha <= 10
    assert min(t[(2, 3, p, B.OPERAND_TF32, 1)] for p in (1, 2, 3)) <= 700
    assert min(t[(4, 3, p, B.OPERAND_TF32, 1)] for p in (1, 2, 3)) > 700
    assert min(t[(4, 3, p, B.OPERAND_BF16, 3)] for p in (1, 2, 3)) <= 700
    assert min(t[(6, 3, p, B.OPERAND_BF16, 1)] for p in (1, 2, 3)) > 7000


# ---------------------------------------------------------------------------
# The twin against arithmetic done by hand.
# ---------------------------------------------------------------------------
CAL = [100000, 50000, 2000, 1000, 20000, 3000000, 64 << 20, 100, 500000, 50000, 10000, 1000000, 2000000, 0, 0, 0]


def test_kernel_cost_is_the_largest_bound_plus_the_launch_term():
    assert T.kernel_ps(CAL) == 3000000
    assert T.kernel_ps(CAL, mem_as=7 * 10 ** 12) == 7000000 + 3000000
    assert T.kernel_ps(CAL, mem_as=7 * 10 ** 12, tensor_as=9 * 10 ** 12, alu_as=8 * 10 ** 12) == 9000000 + 3000000
    assert T.kernel_ps(CAL, mem_as=1999999) == 1 + 3000000           # truncating division
    assert T.kernel_ps(CAL, mem_as=2 ** 200) == T.SATURATED


def test_direct_cost_by_hand():
    # 1 image, 2 -> 3 channels, 4 x 4, k = 3, pad 1: 4 x 4 outputs
    L = T.Layer(1, 2, 3, 4, 4, 3, 1, 1)
    traffic = 4 * (2 * 16 + 3 * 16 + 3 * 2 * 9)            # 536 bytes
    flops = 2 * 3 * 2 * 16 * 9                              # 1728
    # two input channels: twice the few-channel rate constant c[9] (c[9] itself is the 3 -> Cout 3x3 stride-2 kernel's)
    assert T.direct_cost(L, CAL) == max(traffic * 100000, flops * 2 * 50000) // 10 ** 6 + 3000000
    Ls = T.Layer(2, 3, 32, 8, 8, 3, 2, 1)                   # that kernel's shape: 4 x 4 outputs
    tr = 4 * (2 * 3 * 64 + 2 * 32 * 16 + 32 * 27)
    fl = 2 * 2 * 32 * 3 * 16 * 9
    assert T.direct_cost(Ls, CAL) == max(tr * 100000, fl * 50000) // 10 ** 6 + 3000000
    assert T.direct_cost(T.Layer(2, 3, 32, 8, 8, 3, 1, 1), CAL) > 0 and \
        T.direct_cost(T.Layer(2, 3, 32, 8, 6, 3, 2, 1), CAL) == \
        max(4 * (2 * 3 * 48 + 2 * 32 * 12 + 32 * 27) * 100000, 2 * 2 * 32 * 3 * 12 * 9 * 2 * 50000) // 10 ** 6 + 3000000
    L8 = T.Layer(1, 8, 3, 4, 4, 3, 1, 1)
    assert T.direct_cost(L8, CAL) == max(4 * (8 * 16 + 48 + 3 * 8 * 9) * 100000, 2 * 3 * 8 * 16 * 9 * 500000) // 10 ** 6 + 3000000


def test_winograd_cost_by_hand():
    # 2 images, 8 -> 16 channels, 8 x 8, k = 3, pad 1, m = 2, TF32 x1: alpha 4, 16 tiles per image
    L = T.Layer(2, 8, 16, 8, 8, 3, 1, 1)
    chunk, n_chunks, cost = T.winograd_cost(L, 2, T.OPERAND_TF32, 1, CAL)
    assert (chunk, n_chunks) == (2, 1)
    v = 2 * 16 * 16 * 8 * 4
    mm = 2 * 16 * 16 * 16 * 4
    u = 16 * 16 * 8 * 4
    x = 4 * 2 * 8 * 64
    y = 4 * 2 * 16 * 64
    t_in = max(x * 100000 + v * 50000, 4 * 4 * 16 * 2 * 16 * 8 * 20000) // 10 ** 6 + 3000000
    t_con = max((v + mm) * 50000 + u * 100000, 2 * 16 * 16 * 8 * 2 * 16 * 2000) // 10 ** 6 + 3000000
    t_out = max(mm * 50000 + y * 100000, 2 * 2 * 4 * 6 * 2 * 16 * 16 * 20000) // 10 ** 6 + 3000000
    assert cost == t_in + t_con + t_out


def test_winograd_rounds_and_large_tiles_by_hand():
    """The contraction's tensor time counts full rounds of work items over the SMs, and the input transform's
    ALU term grows with alpha in the measured steps (quarters 4, 8, 9, 16).  Constants chosen so that the
    tensor and ALU terms decide: memory free, 1e9 as per tensor flop, 1e9 as per ALU flop, 7 SMs."""
    cal = [0, 0, 10 ** 9, 10 ** 9, 10 ** 9, 1000, 1 << 40, 7, 1, 1, 0, 0, 0, 0, 0, 0]
    # 1 image, 8 -> 16 channels, 4 x 4 outputs, m = 2: alpha 4, 4 tiles: 1 tile block x 1 channel block x 16
    # positions = 16 items on 7 SMs = 3 rounds
    L = T.Layer(1, 8, 16, 4, 4, 3, 1, 1)
    _, _, cost = T.winograd_cost(L, 2, T.OPERAND_TF32, 1, cal)
    flops_con = 2 * 16 * 16 * 8 * 4
    t_con = (flops_con * 10 ** 9 // 16 * 21) // 10 ** 6 + 1000
    t_in = (4 * 4 * 16 * 4 * 8 * 10 ** 9) // 10 ** 6 + 1000
    t_out = (2 * 2 * 4 * 6 * 4 * 16 * 10 ** 9) // 10 ** 6 + 1000
    assert cost == t_in + t_con + t_out
    # the same layer with 7 x 7 kernels: m = 2 -> alpha 8 (8 quarters), m = 4 -> alpha 10 (9), m = 6 -> alpha 12 (16)
    L7 = T.Layer(1, 8, 16, 12, 12, 7, 1, 3)
    for m, quarters in ((2, 8), (4, 9), (6, 16)):
        alpha = m + 6
        tiles = (12 // m) ** 2
        _, _, cost = T.winograd_cost(L7, m, T.OPERAND_TF32, 1, cal)
        items = alpha * alpha                              # 1 tile block, 1 channel block
        rounds_sms = -(-items // 7) * 7
        t_in = (quarters * alpha * alpha * alpha * tiles * 8 * 10 ** 9) // 10 ** 6 + 1000
        t_con = (2 * alpha * alpha * 16 * 8 * tiles * 10 ** 9 // items * rounds_sms) // 10 ** 6 + 1000
        t_out = (2 * m * alpha * (alpha + m) * tiles * 16 * 10 ** 9) // 10 ** 6 + 1000
        assert cost == t_in + t_con + t_out, m


def test_fused_cost_by_hand():
    L = T.Layer(2, 64, 256, 8, 8, 3, 1, 1)                 # 32 tiles: 1 tile block, 2 channel blocks, 2 K blocks
    x, y, u = 4 * 2 * 64 * 64, 4 * 2 * 256 * 64, 16 * 256 * 64 * 4
    block = max(16 * 128 * 32 * 4 * 10000 // 10 ** 6, 1000000)
    serial = 1 * (2 * block + 2000000)
    assert T.fused_cost(L, CAL) == max((x + y + u) * 100000 + x * 50000, serial * 10 ** 6) // 10 ** 6 + 3000000


def test_contraction_tiling_by_hand():
    assert T.contraction_tiling(10, 36, 512, 148) == (256, 2)
    assert T.contraction_tiling(1, 1, 64, 148) in ((64, 1), (32, 2), (16, 4))
    bn, blocks = T.contraction_tiling(98, 36, 24, 148)
    assert bn % 16 == 0 and bn * blocks >= 24


# One output channel: the direct kernel is a thread per output there and may not be booked at the tile kernel's rate (measured
# 545 us against Winograd's 134, 474 / 144, 77 / 32); from two channels on it is the tile kernel.
@pytest.mark.parametrize("shape,direct", [((5, 448, 1, 63, 167, 2, 1, 0), False), ((15, 128, 1, 120, 120, 3, 1, 1), False),
                                          ((7, 43, 1, 150, 25, 3, 1, 3), False), ((1, 24, 40, 33, 31, 3, 1, 1), True)])
def test_one_output_channel_is_not_booked_as_tiles(shape, direct):
    info = compare(W.ConvLayer("one", *shape), {}, {}, B.mnn_get_calibration())
    assert (info.algo == B.ALGO_DIRECT) == direct


def test_direct_cost_of_short_patches_by_hand():
    L = T.Layer(1, 32, 32, 28, 28, 3, 1, 1)                 # 288 patch elements, 14.45 Mflop, 0.24 MB
    flops, traffic = 2 * 32 * 32 * 784 * 9, 4 * (32 * 784 * 2 + 32 * 32 * 9)
    by_patch, by_rate = 288 * 13300000000 + flops * 571000 * 3 // 10, flops * 571000
    cal = list(CAL)
    cal[0], cal[5], cal[8] = 173000, 3530000, 571000
    assert by_patch < by_rate and traffic * 173000 < by_patch
    assert T.direct_cost(L, cal) == by_patch // 10 ** 6 + 3530000
    one = T.Layer(1, 32, 1, 28, 28, 3, 1, 1)
    assert T.direct_cost(one, cal) == 2 * 32 * 784 * 9 * 571000 // 10 ** 6 + 3530000


def test_packed_line_tiling_by_hand():
    # 64 -> 32 channels 3x3 at 9 x 9, one image, BF16: one plane, cells of pitch 10 (one zero column shared by neighbouring
    # rows), taps at 0..22 rows, 100 cells + 22 positions of 128 bytes; one item of 128 cells x 32 channels, three taps a step
    p = T.packed_lines(T.Layer(1, 64, 32, 9, 9, 3, 1, 1), T.OPERAND_BF16, 148)
    issue = 3 * 194000 + 9 * 4 * 45000                      # three steps, 36 instructions
    mma, load = 9 * 4 * (212 * 32 + 15000), (9 * 32 * 128 + 152 * 128) * 63 // 5
    drain = 32 * 512 * 28 + 1087000
    assert issue > mma and issue > load
    assert (p["a_bytes"], p["bn"], p["mt"], p["g"], p["few"]) == (122 * 128, 32, 1, 3, False)
    assert p["product_ps"] == issue + 285000 + 363000 + drain
    # 3 channels 7x7 stride 2 at 224 x 224: kernel columns among the elements, two row phases, seven strips of 16 columns
    q = T.packed_lines(T.Layer(1, 3, 64, 224, 224, 7, 2, 3), T.OPERAND_TF32, 148)
    assert q["few"] and q["width"] == 16 and q["a_bytes"] % (2 * 128) == 0
    assert q["a_bytes"] // 256 >= 7 * 16 * 112              # a position per cell and phase at least


def test_k_loop_splits_by_hand():
    # doubled while twice the CTAs fit the SMs and each keeps four blocks: 10 items 10 -> 20 -> 40 of 148; 32 blocks allow 8
    assert [T.cluster_split(10, k, 148) for k in (7, 8, 15, 16, 32, 100)] == [1, 2, 2, 4, 4, 4]
    assert [T.cluster_split(8, k, 148) for k in (31, 32)] == [4, 8]
    assert [T.cluster_split(n, 64, 148) for n in (18, 19, 37, 38, 74, 75)] == [4, 4, 4, 2, 2, 1]
    # the contraction: not below 20 blocks, in two not below 36
    assert [T.tile_copy_split(10, k, 148) for k in (8, 19, 20, 64)] == [1, 1, 4, 4]
    assert [T.tile_copy_split(50, k, 148) for k in (20, 35, 36)] == [1, 1, 2]


def test_first_minimum_wins_ties_and_inadmissible_is_never_chosen():
    L = T.Layer(32, 128, 128, 28, 28, 3, 1, 1)
    ppm = {key: 1 for key in ppm_table()}                   # everything admissible
    ch = T.plan(L, T.Options(), CAL, ppm)
    assert ch.cost_ps[ch.chosen] == min(ch.cost_ps)
    assert ch.chosen == ch.cost_ps.index(min(ch.cost_ps))
    ppm_bad = {key: 10 ** 9 for key in ppm}                 # nothing with rounding is admissible: only direct remains
    ch = T.plan(L, T.Options(), CAL, ppm_bad)
    assert ch.algo == T.ALGO_DIRECT and all(c == T.INADMISSIBLE for c in ch.cost_ps[1:])


# Few-channel packed lines cut a row into equal strips, together up to strips - 1 columns wider than the row: just below the
# 4 GiB bound of the packed planes the tiling must not find fewer bytes than the choice counted (the plan would fail).
@pytest.mark.parametrize("Cin,k,OW", [(3, 2, 49), (3, 2, 113), (4, 3, 113), (10, 3, 49)])
def test_every_layer_near_the_packed_bound_plans(Cin, k, OW):
    strips = -(-OW // 16)
    at_bound = (4 << 30) // (128 * (OW + k - 1) * max(OW + k - 1, strips * -(-OW // strips)))
    seen = set()
    for N in range(at_bound - 8, int(at_bound * 1.08), max(1, at_bound // 200)):
        layer = W.ConvLayer("near", N, Cin, 4, OW + k - 1, OW + k - 1, k, 1, 0, relu=False)
        info = compare(layer, dict(force_algo=B.ALGO_GEMM, operand=B.OPERAND_TF32, passes=1),
                       dict(force_algo=T.ALGO_GEMM, operand=T.OPERAND_TF32, passes=1), B.mnn_get_calibration())
        seen.add(info.gemm_lhs == B.GEMM_LHS_PACKED)
    assert seen == {True, False}


# Layers whose K loop is cut over clusters: the implicit gather where its serial gather is the shorter way (ResNet-18's
# stride-2 layers at one image), the patch matrix where it is not (measured 67 against 100, 63 / 96, 259 / 425, 46 / 57 us).
@pytest.mark.parametrize("shape,lhs", [
    ((1, 64, 128, 56, 56, 3, 2, 1, 1), B.GEMM_LHS_IMPLICIT), ((1, 128, 256, 28, 28, 3, 2, 1, 1), B.GEMM_LHS_IMPLICIT),
    ((1, 256, 512, 14, 14, 3, 2, 1, 1), B.GEMM_LHS_IMPLICIT), ((47, 304, 304, 8, 8, 3, 2, 1, 1), B.GEMM_LHS_PATCHES),
    ((19, 107, 134, 9, 37, 5, 2, 2, 1), B.GEMM_LHS_PATCHES), ((16, 383, 365, 17, 100, 6, 2, 0, 3), B.GEMM_LHS_PATCHES),
    ((6, 31, 174, 15, 15, 7, 1, 12, 4), B.GEMM_LHS_PATCHES)])
def test_cut_layers_take_the_shorter_gather(shape, lhs):
    N, Cin, Cout, H, W_, k, stride, pad, dil = shape
    layer = W.ConvLayer("cut", N, Cin, Cout, H, W_, k, stride, pad, dil)
    if k == 6:                                               # (no accuracy figures for this size in the table)
        plan = B.mnn_conv_plan_ex(*shape, B.make_opts(relu=1))
        info = B.mnn_conv_plan_query(plan)
        B.mnn_conv_destroy(plan)
    else:
        info = compare(layer, {}, {}, B.mnn_get_calibration())
    assert (info.algo, info.gemm_lhs) == (B.ALGO_GEMM, lhs)


def test_the_gathers_choice_does_not_depend_on_its_booked_rate(restore_calibration):
    # the gather's pace is a figure of the kernel: with the rate that calibration finds (250e6 against the built-in 400e6) the
    # booked costs move, but where the patch matrix is still booked the choice between the two must stay
    l = W.ConvLayer("cut", 47, 304, 304, 8, 8, 3, 2, 1, 1)
    kw = dict(force_algo=B.ALGO_GEMM, operand=B.OPERAND_TF32, passes=1)
    for rate in (400, 250):
        cal = list(restore_calibration)
        cal[13] = rate * 10 ** 6
        B.mnn_set_calibration(cal)
        assert compare(l, kw, kw, cal).gemm_lhs == B.GEMM_LHS_PATCHES


# Packed lines against the operand they replace, each by its own time (measured 196 against 595 us, 52 / 104, 56 / 133, 402 / 1183,
# 290 / 595 where the lines lose; 53 / 27, 86 / 37 where they win).
@pytest.mark.parametrize("shape,packed", [
    ((30, 256, 348, 26, 26, 7, 1, 1, 4), False), ((36, 2, 289, 60, 60, 5, 1, 2, 1), False),
    ((26, 2, 419, 146, 59, 7, 1, 0, 1), False), ((47, 416, 406, 5, 168, 5, 2, 5, 3), False), ((16, 3, 326, 172, 172, 3, 1, 0, 1), False),
    ((32, 64, 128, 56, 56, 3, 2, 1, 1), True), ((16, 256, 256, 28, 28, 3, 1, 2, 2), True), ((32, 3, 64, 224, 224, 7, 2, 3, 1), True)])
def test_packed_lines_are_compared_by_their_own_time(shape, packed):
    N, Cin, Cout, H, W_, k, stride, pad, dil = shape
    kw = dict(force_algo=B.ALGO_GEMM, operand=B.OPERAND_TF32, passes=1)
    info = compare(W.ConvLayer("lines", N, Cin, Cout, H, W_, k, stride, pad, dil), kw, kw, B.mnn_get_calibration())
    assert (info.gemm_lhs == B.GEMM_LHS_PACKED) == packed


# Layers on the GEMM scheme: row-wise Winograd (the first), or F(2, 3) by rows, is estimated faster there, but would spread an infinity
# over its tiles, and the first would need 47 MB of workspace instead of 6.
@pytest.mark.parametrize("shape", [(43, 32, 240, 120, 5, 7, 1), (26, 48, 1552, 70, 2, 3, 1), (5, 16, 128, 83, 22, 3, 1), (26, 16, 1408, 12, 12, 3, 0)])
def test_winograd_by_rows_replaces_winograd_only(shape):
    N, Cin, Cout, H, W_, k, pad = shape
    info = compare(W.ConvLayer("gemm", N, Cin, Cout, H, W_, k, 1, pad), {}, {}, B.mnn_get_calibration())
    assert info.algo == B.ALGO_GEMM and info.workspace_bytes <= B.STATIC_WORKSPACE_BYTES


def test_the_gpu_tests_reach_every_kernel_by_rows():
    from tests.test_gpu_rows import SHAPES
    got = set()
    for s, expected in SHAPES:
        if "wise" not in expected:
            t = T.rows_tiling(T.Layer(*s[:6], 1, s[6], 1, 1), 2 if expected == "rows2" else 1, 1 if expected == "bf16" else 3, 148)
            got.add((expected == "rows2", s[5], t["mode"], "two tiles" if t["mt"] == 2 else "cluster" if t["split"] > 1 else "one tile"))
    want = {(False, k, mode, form) for k in (2, 3, 5, 7) for mode in (1, 2, 3) for form in ("one tile", "two tiles", "cluster")}
    want -= {(False, 5, 3, "cluster"), (False, 7, 3, "cluster"), (False, 7, 3, "one tile")}      # not compiled
    assert got == want | {(True, 3, 3, "one tile"), (True, 3, 3, "cluster")}


# Few items share their stages out over clusters, unevenly too (7 over 4): cut in two only, the first two lost to three Winograd kernels.
@pytest.mark.parametrize("shape,precision,split", [((1, 112, 112, 10, 10, 3, 1), B.PREC_TF32, 4), ((2, 111, 111, 9, 9, 3, 1), B.PREC_BF16, 4),
                                                   ((4, 96, 96, 5, 7, 3, 1), B.PREC_TF32, 4), ((1, 178, 178, 10, 10, 3, 1), B.PREC_BF16, 8),
                                                   ((1, 64, 100, 11, 10, 3, 1), B.PREC_TF32, 1)])
def test_rows_share_their_stages_unevenly(shape, precision, split):
    N, Cin, Cout, H, W_, k, pad = shape
    info = compare(W.ConvLayer("split", N, Cin, Cout, H, W_, k, 1, pad), dict(precision=precision), dict(precision=precision), B.mnn_get_calibration())
    assert info.gemm_lhs == B.GEMM_LHS_ROWS
    t = T.rows_tiling(T.Layer(N, Cin, Cout, H, W_, k, 1, pad, 1), 1, 3 if precision == B.PREC_TF32 else 1, 148)
    assert t["split"] == split


# Packed lines against the convolution by rows, at the sizes where either was measured faster by more than 4 % (us in lines and by rows):
# neither the number of output channels nor the accuracy class decides alone.
@pytest.mark.parametrize("shape,precision,rows", [
    ((64, 256, 96, 56, 56, 3, 1), B.PREC_BF16, False),      # 155, 188
    ((64, 256, 192, 56, 56, 3, 1), B.PREC_BF16, True),      # 226, 203
    ((64, 256, 255, 56, 56, 3, 1), B.PREC_BF16, True),      # 252, 242
    ((64, 256, 256, 56, 56, 3, 1), B.PREC_BF16, True),      # 244, 237 (262 and 302 call after call)
    ((64, 256, 288, 56, 56, 3, 1), B.PREC_BF16, False),     # 295, 399
    ((10, 256, 256, 95, 95, 3, 1), B.PREC_BF16, False),     # 124, 158
    ((18, 64, 160, 28, 28, 3, 1), B.PREC_BF16, True),       # 12.5, 9.7
    ((4, 192, 464, 26, 26, 2, 1), B.PREC_BF16, False),      # 11.1, 13.6
    ((5, 64, 400, 15, 9, 3, 1), B.PREC_BF16, False),        # 6.3, 7.0
    ((13, 6, 181, 62, 41, 3, 1), B.PREC_TF32, True)])       # 18.5, 11.9
def test_rows_against_packed_lines(shape, precision, rows):
    N, Cin, Cout, H, W_, k, pad = shape
    info = compare(W.ConvLayer("lines", N, Cin, Cout, H, W_, k, 1, pad), dict(precision=precision), dict(precision=precision), B.mnn_get_calibration())
    assert (info.gemm_lhs == B.GEMM_LHS_ROWS) == rows


def test_routing_rules():
    t = ppm_table()
    for l in all_layers():
        ch = T.plan(twin_layer(l), T.Options(), CAL, t)
        if l.k == 1:
            assert ch.algo != T.ALGO_WINOGRAD                # k = 1 "is just a matrix multiplication"
        if l.stride > 1 or l.dilation > 1 or l.groups > 1:
            assert ch.algo != T.ALGO_WINOGRAD
        if l.groups > 1:
            assert ch.algo == T.ALGO_DIRECT
    # cost never decreases with the batch
    for n in (1, 2, 4, 8, 16, 32, 64):
        a = T.plan(T.Layer(n, 64, 64, 56, 56, 3, 1, 1), T.Options(), CAL, t)
        b = T.plan(T.Layer(2 * n, 64, 64, 56, 56, 3, 1, 1), T.Options(), CAL, t)
        assert all(x <= y for x, y in zip(a.cost_ps, b.cost_ps))


def test_paper_count_on_a_worked_example():
    # Eq. 2 with o_c on its third term, times the tiles: 1 -> 1 channel, 4 x 4 input, k = 3, no padding: 2 x 2 outputs
    L = T.Layer(1, 1, 1, 4, 4, 3, 1, 0)
    assert T.paper_multiplications(L, 2) == 1 * (2 * 64 + 16 + 2 * 4 * 6)          # one 4 x 4 tile
    assert T.paper_multiplications(L, 1) == 4 * (2 * 27 + 9 + 1 * 3 * 4)           # four 3 x 3 "tiles"
    assert T.paper_choice(L)[0] == 2
    # many channels: the Hadamard term i_c o_c alpha^2 per tile dominates and the largest tile wins
    assert T.paper_choice(T.Layer(1, 512, 512, 48, 48, 3, 1, 1))[0] == 6     # 64 tiles x 64 < 144 x 36 < 576 x 16
