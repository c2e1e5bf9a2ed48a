"""The convolution by rows in one kernel (rows_conv.cu) and row-wise Winograd (line_wino.cu) on the GPU, as the planner chooses them,
against the fp64 oracle: last tiles and channel blocks that are not full, padded channels, odd rows, paddings other than the one that
keeps the size, every kernel size, clusters, both accuracy classes; integer inputs bit for bit; repeated runs; NaN."""
import numpy as np
import pytest

from oracle import direct_conv as oc
from paper_2002_12418_b200 import binding as B
from paper_2002_12418_b200 import workloads as W
from tests.util import rel_l2, to_dev

pytestmark = pytest.mark.gpu

# The planner's own figures where it admits a form by them: F(2, 3) by rows 8 ppm, row-wise F(4, 5) and F(2, 7) 30, F(4, 3) 20.  The
# definition: hi + lo BF16 operands leave 2^-17 of each factor and drop lo * lo, 3 * 2^-17 = 2.3e-5 of a product at most, as a 2-norm over
# many terms of random sign a fifth of that (predicted 4 to 5 ppm; 7 with one output channel), so 1e-5.  One BF16 product: 2 * 2^-9.
BOUND = {"rows1": 1e-5, "rows2": 8e-6, "wise": 3e-5, "wise3": 2e-5, "bf16": 4e-3}


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available()
    B.lib()
    return torch


def form(info):
    if info.algo == B.ALGO_GEMM and info.gemm_lhs == B.GEMM_LHS_ROWS:
        return "rows1" if info.passes == 3 else "bf16"
    return {B.FUSED_BY_ROWS: "rows2", B.ROW_WISE: "wise"}.get(info.fused) if info.algo == B.ALGO_WINOGRAD else None


def run(torch, shape, x, w, b, relu, cls=B.PREC_TF32, repeats=1):
    N, Cin, Cout, H, W_, k, pad = shape
    r = B.ConvLayerRunner(N, Cin, Cout, H, W_, k, 1, pad, 1, B.make_opts(relu=relu, precision=cls))
    info = r.info
    xd, wd, bd = to_dev(torch, x), to_dev(torch, w), to_dev(torch, b) if b is not None else None
    ys = []
    for _ in range(repeats):
        y = torch.full((N, Cout, info.OH, info.OW), float("nan"), device="cuda:0")
        r.run(xd, wd, bd, y)
        ys.append(y)
    torch.cuda.synchronize()
    assert r.device_status() == 0
    r.close()
    assert all(torch.equal(ys[0], y) for y in ys[1:])
    return ys[0].cpu().numpy(), info


# (N, Cin, Cout, H, W, k, pad); a shape at least per instantiation of the kernel by rows (kernel size, products and how they are issued, one or
# two tiles per item or clusters: tests/test_planner_twin.py checks that), row-wise with one and several channel blocks, full and not, and
# scalar, 64-bit and 128-bit loads; paddings up to more than k - 1, up to 841 input channels
SHAPES = [((2, 100, 33, 8, 26, 2, 1), "rows1"), ((5, 130, 8, 26, 34, 2, 0), "rows1"), ((1, 200, 130, 8, 6, 2, 1), "rows1"), ((1, 256, 8, 26, 29, 2, 1), "rows1"),
          ((17, 16, 17, 33, 39, 2, 1), "rows1"), 
          ((1, 64, 100, 11, 10, 3, 1), "rows1"), ((9, 130, 1, 22, 30, 3, 2), "rows1"), ((1, 130, 64, 5, 17, 3, 1), "rows1"), ((2, 256, 33, 8, 9, 3, 0), "rows1"),
          ((17, 64, 1, 25, 40, 3, 2), "rows1"), ((5, 16, 100, 6, 29, 3, 1), "rows1"), ((1, 256, 130, 11, 5, 3, 0), "rows1"),
          ((17, 16, 8, 30, 38, 3, 1), "rows1"), ((7, 100, 72, 35, 45, 3, 1), "rows1"),
          ((1, 16, 200, 8, 10, 5, 2), "rows1"), ((9, 64, 1, 38, 18, 5, 2), "rows1"), ((5, 130, 1, 12, 33, 5, 4), "rows1"), ((17, 24, 1, 36, 29, 5, 2), "rows1"),
          ((17, 16, 33, 36, 20, 5, 0), "rows1"), ((1, 16, 33, 31, 8, 7, 3), "rows1"), ((5, 64, 1, 34, 20, 7, 3), "rows1"), ((2, 256, 1, 5, 34, 7, 6), "rows1"),
          ((17, 17, 1, 25, 37, 7, 6), "rows1"),
          ((2, 100, 33, 34, 6, 2, 1), "bf16"), ((1, 33, 100, 23, 9, 3, 1), "bf16"), ((1, 130, 33, 15, 11, 3, 1), "bf16"), ((3, 256, 8, 19, 9, 3, 0), "bf16"),
          ((9, 130, 1, 28, 29, 3, 1), "bf16"), ((2, 17, 100, 27, 7, 5, 0), "bf16"), ((1, 256, 1, 39, 35, 5, 4), "bf16"), ((17, 130, 1, 34, 36, 5, 4), "bf16"),
          ((1, 24, 72, 6, 13, 7, 3), "bf16"), ((1, 256, 64, 15, 12, 7, 0), "bf16"),
          ((32, 64, 64, 56, 56, 3, 1), "rows2"), ((17, 17, 17, 29, 37, 3, 1), "rows2"), ((17, 130, 1, 39, 30, 3, 0), "rows2"), ((17, 256, 1, 9, 33, 3, 1), "rows2"),
          ((1, 256, 8, 37, 30, 3, 0), "rows2"), 
          # 3, 7, 12 and 13 stages shared out unevenly over clusters
          ((8, 44, 16, 12, 19, 7, 6), "rows1"), ((1, 112, 100, 10, 10, 3, 1), "rows1"), ((1, 186, 40, 10, 10, 3, 1), "rows1"), ((2, 200, 100, 6, 5, 3, 1), "bf16"),
          ((17, 256, 1, 33, 31, 5, 2), "wise"), ((17, 256, 1, 18, 9, 7, 3), "wise"), ((17, 130, 1, 33, 38, 7, 0), "wise"), ((64, 128, 128, 28, 28, 5, 2), "wise"),
          ((39, 72, 17, 8, 4, 2, 1), "bf16"), ((19, 66, 56, 6, 5, 2, 1), "rows1"), ((36, 22, 1, 65, 45, 2, 1), "bf16"), ((5, 105, 57, 8, 5, 2, 1), "bf16"), ((2, 78, 10, 17, 108, 2, 0), "rows1"), ((39, 70, 1, 34, 31, 2, 0), "rows1"),
          ((2, 186, 7, 7, 117, 2, 0), "rows1"), ((43, 26, 1, 37, 24, 3, 2), "bf16"), ((10, 8, 18, 51, 36, 3, 2), "rows1"), ((6, 45, 2, 16, 103, 3, 2), "rows1"),
          ((2, 104, 6, 5, 94, 3, 2), "rows1"), ((21, 5, 68, 70, 9, 5, 4), "rows1"), ((5, 3, 264, 95, 5, 5, 4), "rows1"), ((55, 6, 8, 11, 45, 7, 0), "bf16"),
          ((29, 6, 83, 7, 62, 7, 6), "rows1"), ((1, 512, 64, 7, 7, 3, 1), "rows1"), ((2, 40, 33, 12, 10, 5, 6), "rows1"), ((2, 48, 33, 14, 10, 3, 3), "rows1"),
          ((28, 791, 1, 7, 21, 3, 4), "wise3"), ((16, 841, 667, 4, 6, 3, 4), "wise3"), ((7, 469, 29, 5, 39, 5, 6), "wise"), ((18, 323, 1, 14, 32, 5, 2), "wise"),
          ((28, 59, 692, 14, 20, 5, 2), "wise"), ((5, 316, 434, 4, 4, 7, 8), "wise"), ((23, 160, 1, 10, 14, 7, 3), "wise"), ((22, 319, 136, 14, 6, 7, 3), "wise")]


@pytest.mark.parametrize("shape,expected", SHAPES)
def test_against_the_oracle(torch, shape, expected):
    N, Cin, Cout, H, W_, k, pad = shape
    layer = W.ConvLayer("rows", N, Cin, Cout, H, W_, k, 1, pad, relu=True, seed=sum(shape))
    x, w, b = W.make_inputs(layer)
    cls = B.PREC_BF16 if expected == "bf16" else B.PREC_TF32
    got, info = run(torch, shape, x, w, b, True, cls, repeats=3)
    assert form(info) == expected.rstrip("3")
    assert info.predicted_error_ppm * 1e-6 <= BOUND[expected]
    assert rel_l2(got, oc.direct_conv(x, w, b, 1, pad, 1, 1, True)) <= BOUND[expected]


# 1 x k and k x 1 kernels left to the plan take the same kernel: every kernel size, one tile and two per item, clusters, odd paddings.
@pytest.mark.parametrize("N,Cin,Cout,H,W_,kh,kw,ph,pw", [
    (9, 82, 82, 25, 17, 1, 3, 0, 1), (32, 192, 192, 17, 17, 1, 7, 0, 3), (32, 192, 192, 17, 17, 7, 1, 3, 0), (1, 33, 33, 31, 34, 1, 7, 2, 5),
    (6, 36, 211, 31, 24, 5, 1, 2, 3), (4, 50, 203, 20, 18, 3, 1, 0, 1), (35, 112, 58, 14, 27, 1, 5, 0, 2), (3, 40, 17, 12, 33, 1, 2, 0, 1), (3, 40, 17, 33, 12, 2, 1, 1, 0)])
def test_line_kernels(torch, N, Cin, Cout, H, W_, kh, kw, ph, pw):
    rng = np.random.Generator(np.random.PCG64(N + Cin + kh))
    x = np.maximum(rng.standard_normal((N, Cin, H, W_), dtype=np.float32), 0)
    w = (rng.standard_normal((Cout, Cin, kh, kw)) * np.sqrt(2.0 / (Cin * kh * kw))).astype(np.float32)
    b = (rng.standard_normal((Cout,)) * 0.1).astype(np.float32)
    r = B.ConvLayerRunner(N, Cin, Cout, H, W_, max(kh, kw), plan=B.mnn_conv_plan_rect(N, Cin, Cout, H, W_, kh, kw, ph, pw, B.make_opts(relu=1)))
    assert form(r.info) == "rows1"
    y = r.run(to_dev(torch, x), to_dev(torch, w), to_dev(torch, b))
    torch.cuda.synchronize()
    assert r.device_status() == 0
    r.close()
    assert rel_l2(y.cpu().numpy(), oc.direct_conv_rect(x, w, b, ph, pw, True)) <= BOUND["rows1"]


# Small integers are exact in BF16 and in fp32 sums: the definition bit for bit.
@pytest.mark.parametrize("shape", [(5, 16, 100, 6, 29, 3, 1), (2, 256, 33, 8, 9, 3, 0), (17, 24, 1, 36, 29, 5, 2)])
def test_integers_bit_for_bit(torch, shape):
    N, Cin, Cout, H, W_, k, pad = shape
    rng = np.random.Generator(np.random.PCG64(7))
    x, w, b = (rng.integers(-3, 4, size=s).astype(np.float32) for s in ((N, Cin, H, W_), (Cout, Cin, k, k), (Cout,)))
    got, info = run(torch, shape, x, w, b, False)
    assert form(info) == "rows1"
    assert np.array_equal(got.astype(np.float64), oc.direct_conv(x, w, b, 1, pad, 1, 1, False))


# What is no number stays where its windows reach, without ReLU too.
def test_not_a_number_reaches_its_windows_only(torch):
    shape = (1, 64, 100, 11, 10, 3, 1)
    N, Cin, Cout, H, W_, k, pad = shape
    x, w, _ = W.make_inputs(W.ConvLayer("nan", N, Cin, Cout, H, W_, k, 1, pad, seed=5))
    clean, _ = run(torch, shape, x, w, None, False)
    x[0, 7, 4, 5] = np.nan
    got, info = run(torch, shape, x, w, None, False)
    assert form(info) == "rows1"
    near = np.zeros((H, W_), dtype=bool)
    near[3:6, 4:7] = True
    assert np.isnan(got[..., near]).all() and np.array_equal(got[..., ~near], clean[..., ~near])


# Infinite inputs and weights, and inputs that BF16 rounds to infinity, give what the definition gives (with ReLU: fmax(no number, 0)
# is 0), as the TF32 product does; nothing else changes.  One shape per tiles per item and way of issuing the products, one cluster.
@pytest.mark.parametrize("relu", [False, True])
@pytest.mark.parametrize("shape", [(1, 64, 100, 11, 10, 3, 1), (2, 100, 33, 8, 26, 2, 1), (17, 16, 17, 33, 39, 2, 1), (17, 16, 8, 30, 38, 3, 1),
                                   (2, 256, 33, 8, 9, 3, 0)])
def test_infinite_and_largest_values(torch, shape, relu):
    N, Cin, Cout, H, W_, k, pad = shape
    x, w, b = W.make_inputs(W.ConvLayer("inf", N, Cin, Cout, H, W_, k, 1, pad, seed=6))
    x[:, 1] *= 0.2                                       # (no product with the largest weight may pass the largest number in one sum and not in the other)
    clean, info = run(torch, shape, x, w, b, relu)
    assert form(info) == "rows1"
    x[0, 7, 4, 5], x[0, 3, 1, 1], x[N - 1, Cin - 1, H - 1, 0] = np.inf, -np.inf, 3.4e38
    w[2, 5, 0, 0], w[4, 1, 1, 1] = np.inf, 3.4e38
    got, _ = run(torch, shape, x, w, b, relu)
    _check_not_finite(got, clean, oc.direct_conv(x, w, b, 1, pad, 1, 1, False), relu, [2, 4])


@pytest.mark.parametrize("N,Cin,Cout,H,W_,kh,kw,ph,pw", [(3, 40, 17, 12, 33, 1, 2, 0, 1), (6, 36, 211, 31, 24, 5, 1, 2, 3), (2, 40, 24, 61, 1, 3, 1, 1, 0)])
def test_infinite_and_largest_values_line_kernels(torch, N, Cin, Cout, H, W_, kh, kw, ph, pw):
    rng = np.random.Generator(np.random.PCG64(8))
    x = rng.standard_normal((N, Cin, H, W_), dtype=np.float32)
    w = (rng.standard_normal((Cout, Cin, kh, kw)) * 0.1).astype(np.float32)
    outs = []
    for special in (False, True):
        if special:
            x[0, 7, 4, W_ // 2], x[1, 3, 1, 0], x[N - 1, Cin - 1, H - 1, 0] = np.inf, -np.inf, 3.4e38
        r = B.ConvLayerRunner(N, Cin, Cout, H, W_, max(kh, kw), plan=B.mnn_conv_plan_rect(N, Cin, Cout, H, W_, kh, kw, ph, pw, B.make_opts()))
        assert form(r.info) == "rows1"
        y = r.run(to_dev(torch, x), to_dev(torch, w), None)
        torch.cuda.synchronize()
        assert r.device_status() == 0
        outs.append(y.cpu().numpy())
        r.close()
    _check_not_finite(outs[1], outs[0], oc.direct_conv_rect(x, w, None, ph, pw, False), False, [])


def _check_not_finite(got, clean, ref, relu, touched_channels):
    """`ref` is the fp64 sum; outputs it leaves at ordinary size are those of the clean run, bit for bit."""
    fp32 = ref.astype(np.float32)                        # beyond the largest fp32 number: infinite
    large = ~(np.abs(ref) < 1e30)
    assert large.any() and np.isinf(fp32).any()
    want = np.where(np.isnan(fp32), np.float32(0), np.maximum(fp32, np.float32(0))) if relu else fp32
    same = ~large
    same[:, touched_channels] = False                    # (a large weight may meet zeros of x only)
    assert np.array_equal(got[same], clean[same])
    infinite = large & ~np.isfinite(want)
    assert np.array_equal(got[infinite], want[infinite], equal_nan=True)
    finite = large & np.isfinite(want)                   # fp32 sums of at most 2304 terms
    assert (np.abs(got[finite].astype(np.float64) - want[finite]) <= 2304 * 2.0 ** -23 * 3.4e38).all() and np.isfinite(got[finite]).all()
