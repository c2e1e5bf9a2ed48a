"""The GEMM scheme on packed lines of positions (strided, dilated and few-channel layers) against the fp64 direct-convolution
oracle, through the C ABI.  The planner takes it by itself; a shape that it routes elsewhere would fail the assertion."""
import numpy as np
import pytest

from oracle import direct_conv as oc
from oracle import planner_twin as T
from paper_2002_12418_b200 import binding as B
from paper_2002_12418_b200 import workloads as W
from tests.util import assert_close, to_dev

pytestmark = pytest.mark.gpu

# (N, Cin, Cout, H, W, k, stride, pad, dilation)
SHAPES = [
    (40, 32, 128, 20, 20, 3, 2, 1, 1),       # one block of channels, four phases
    (64, 64, 130, 15, 13, 3, 2, 1, 1),       # odd extents, output channels off the tile, cells that are no outputs
    (16, 96, 40, 30, 44, 3, 1, 2, 2),        # dilation 2
    (9, 64, 272, 37, 33, 3, 1, 3, 3),        # dilation 3, two channel blocks of a wide layer
    (30, 32, 64, 26, 28, 5, 2, 2, 1),        # 25 taps in four phases
    (60, 32, 48, 60, 60, 3, 3, 0, 1),        # stride 3, one tap per phase, no padding
    (40, 64, 64, 47, 51, 2, 2, 1, 1),        # even kernel
    (6, 3, 64, 96, 100, 7, 2, 3, 1),         # few channels: 21 of 24 elements, strips with a partial last one
    (5, 4, 33, 60, 130, 5, 2, 2, 2),         # few channels, dilation, 20 elements
    (7, 6, 24, 70, 65, 5, 2, 1, 1),          # few channels, 30 of 32 elements
]


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available()
    B.lib()
    return torch


def run(torch, layer, inputs):
    x, w, b = inputs
    r = B.ConvLayerRunner(layer.N, layer.Cin, layer.Cout, layer.H, layer.W, layer.k, layer.stride, layer.pad, layer.dilation,
                          B.make_opts(relu=layer.relu, force_algo=B.ALGO_GEMM, operand=B.OPERAND_TF32, passes=1))
    info = r.info
    assert info.gemm_lhs == B.GEMM_LHS_PACKED and info.launches_per_run == 2
    r.workspace.fill_(0xFF)                   # NaNs wherever a kernel reads what none has written
    B.mnn_conv_set_workspace(r.plan, r._ws_ptr, info.workspace_bytes)
    y = torch.full((layer.N, layer.Cout, info.OH, info.OW), float("nan"), device="cuda:0")
    xd, wd, bd = to_dev(torch, x), to_dev(torch, w), to_dev(torch, b) if b is not None else None
    r.run(xd, wd, bd, y)
    again = r.run(xd, wd, bd)
    torch.cuda.synchronize()
    assert r.device_status() == 0 and torch.equal(y, again)
    out = y.cpu().numpy()
    r.close()
    return out


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("relu", [True, False])
def test_parity(torch, shape, relu):
    N, Cin, Cout, H, W_, k, s, p, d = shape
    layer = W.ConvLayer("lines", N, Cin, Cout, H, W_, k, s, p, d, relu=relu, x_dist="normal", seed=sum(shape),
                        bias_dist="normal0.1" if relu else "zero")
    x, w, b = W.make_inputs(layer)
    assert_close(run(torch, layer, (x, w, b)), oc.direct_conv(x, w, b, s, p, d, 1, relu), B.PREC_TF32, "packed lines")


@pytest.mark.parametrize("shape", SHAPES)
def test_integer_inputs_bit_exact(torch, shape):
    N, Cin, Cout, H, W_, k, s, p, d = shape
    layer = W.ConvLayer("lines", N, Cin, Cout, H, W_, k, s, p, d, relu=False, seed=11)
    x, w, b = W.integer_inputs(layer, -3, 3)
    assert np.array_equal(run(torch, layer, (x, w, b)).astype(np.float64), oc.direct_conv(x, w, b, s, p, d, 1, False))


def test_more_than_the_staged_bias(torch):
    layer = W.ConvLayer("lines", 4, 32, 2100, 20, 20, 3, 2, 1, relu=True, seed=5)
    x, w, b = W.make_inputs(layer)
    assert_close(run(torch, layer, (x, w, b)), oc.direct_conv(x, w, b, 2, 1, 1, 1, True), B.PREC_TF32, "packed lines")


# BF16 operands: blocks of 64 channels; one and several blocks, phases, ragged channel tiles, one and two tiles of cells per
# item, and a layer that leaves the Winograd scheme for this form by itself.  Integers are exact in BF16.
@pytest.mark.parametrize("shape,auto", [((20, 64, 40, 17, 19, 3, 1, 1, 1), False), ((90, 64, 130, 15, 13, 3, 2, 1, 1), False),
                                        ((6, 192, 272, 37, 33, 3, 1, 3, 3), False), ((30, 128, 48, 26, 28, 5, 2, 2, 1), False),
                                        ((40, 64, 64, 47, 51, 2, 2, 1, 1), False), ((64, 64, 64, 56, 56, 3, 1, 1, 1), True)])
def test_bf16(torch, shape, auto):
    N, Cin, Cout, H, W_, k, s, p, d = shape
    layer = W.ConvLayer("lines", N, Cin, Cout, H, W_, k, s, p, d, relu=True, seed=sum(shape))
    r = B.ConvLayerRunner(N, Cin, Cout, H, W_, k, s, p, d,
                          B.make_opts(relu=True, precision=B.PREC_BF16, **({} if auto else dict(force_algo=B.ALGO_GEMM, operand=B.OPERAND_BF16))))
    assert (r.info.algo, r.info.gemm_lhs, r.info.operand) == (B.ALGO_GEMM, B.GEMM_LHS_PACKED, B.OPERAND_BF16)
    r.workspace.fill_(0xFF)                   # NaNs wherever a kernel reads what none has written
    B.mnn_conv_set_workspace(r.plan, r._ws_ptr, r.info.workspace_bytes)
    for exact in (True, False):
        x, w, b = W.integer_inputs(layer, -3, 3) if exact else W.make_inputs(layer)
        wd = to_dev(torch, w)
        r.prepare(wd)
        got = r.run(to_dev(torch, x), wd, to_dev(torch, b))
        torch.cuda.synchronize()
        assert r.device_status() == 0
        ref = oc.direct_conv(x, w, b, s, p, d, 1, True)
        if exact:
            assert np.array_equal(got.cpu().numpy().astype(np.float64), ref)
        else:
            assert_close(got.cpu().numpy(), ref, B.PREC_BF16, "packed lines in BF16")
    r.close()


# Every tiling the planner reaches: one, two and four tiles of 128 cells per item (as many issuing threads), one, two and three
# weight tiles per step (partial groups, other slot sizes), three and four tensor-core steps per block.  The planner's
# integer twin names the tiling, so a shape that comes to another one fails.  Integers: exact.
@pytest.mark.parametrize("shape,bf16,mt,g", [
    ((6, 32, 299, 10, 82, 2, 1, 1, 6), False, 1, 1), ((11, 32, 34, 12, 92, 2, 1, 1, 6), False, 1, 2),
    ((10, 32, 1, 28, 65, 3, 1, 1, 4), False, 2, 1), ((29, 32, 18, 13, 33, 3, 1, 6, 6), False, 2, 2),
    ((40, 32, 1, 13, 93, 2, 1, 1, 3), False, 4, 1), ((32, 32, 26, 20, 52, 3, 1, 2, 2), False, 4, 2),
    ((63, 32, 1, 26, 26, 2, 1, 1, 6), False, 4, 3), ((9, 1, 471, 91, 23, 2, 1, 0, 1), False, 1, 2),
    ((14, 2, 178, 109, 69, 5, 1, 0, 2), False, 4, 2), ((20, 9, 1, 25, 76, 3, 1, 1, 1), False, 4, 3),
    ((17, 64, 72, 33, 68, 6, 2, 0, 6), True, 1, 1), ((1, 64, 75, 34, 78, 6, 2, 0, 6), True, 1, 2),
    ((53, 128, 2, 20, 28, 4, 1, 0, 6), True, 2, 1), ((50, 128, 58, 23, 23, 4, 1, 0, 6), True, 2, 2),
    ((48, 64, 1, 11, 87, 2, 1, 0, 3), True, 4, 1), ((55, 64, 18, 27, 27, 3, 1, 1, 4), True, 4, 2),
    ((23, 64, 1, 110, 17, 2, 1, 0, 4), True, 4, 3)])
def test_every_tiling(torch, shape, bf16, mt, g):
    N, Cin, Cout, H, W_, k, s, p, d = shape
    operand = B.OPERAND_BF16 if bf16 else B.OPERAND_TF32
    tiling = T.packed_lines(T.Layer(N, Cin, Cout, H, W_, k, s, p, d), operand, 148)
    assert (tiling["mt"], tiling["g"]) == (mt, g)
    layer = W.ConvLayer("lines", N, Cin, Cout, H, W_, k, s, p, d, relu=False, seed=sum(shape))
    x, w, b = W.integer_inputs(layer, -3, 3)
    r = B.ConvLayerRunner(*shape, B.make_opts(relu=0, precision=B.PREC_BF16 if bf16 else B.PREC_TF32, force_algo=B.ALGO_GEMM,
                                              operand=operand, passes=1))
    assert r.info.gemm_lhs == B.GEMM_LHS_PACKED
    r.workspace.fill_(0xFF)                   # NaNs wherever a kernel reads what none has written
    B.mnn_conv_set_workspace(r.plan, r._ws_ptr, r.info.workspace_bytes)
    y = torch.full((N, Cout, r.info.OH, r.info.OW), float("nan"), device="cuda:0")
    r.run(to_dev(torch, x), to_dev(torch, w), to_dev(torch, b), y)
    torch.cuda.synchronize()
    assert r.device_status() == 0
    assert np.array_equal(y.cpu().numpy().astype(np.float64), oc.direct_conv(x, w, b, s, p, d, 1, False))
    r.close()
