"""The fully quantized transforms where their staging and stores change form: rows copied in 16-byte
pieces, in pairs or one by one, x that is only 4-byte aligned, group sizes without a register variant,
fp32 input, CTAs that take several work items with one strip buffer and with two, every store variant of the
output transform with CTAs of 64 and of 128 tiles, and codes at ties and next to them."""
import numpy as np
import pytest

from oracle import full_quant as fq
from oracle import oracle as orc
from paper_2412_19867_b200 import binding as b
from tests.gpu_util import make_conv
from paper_2412_19867_b200 import workloads as wl
from paper_2412_19867_b200.workloads import Layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 2])           # elements x is moved off its 16-byte alignment
@pytest.mark.parametrize("layer", [
    Layer(2, 64, 24, 9, 24, 4, 64, "f16", "silu_outlier", "kaiming_chan", 8, 20, 0),     # 16-byte pieces
    Layer(1, 96, 17, 7, 10, 6, 32, "f16", "silu_outlier", "kaiming_chan", 8, 21, 0),     # pairs
    Layer(1, 192, 8, 5, 13, 4, 96, "f16", "relu_heavy", "kaiming", 8, 22, 0),            # single elements, odd W
    Layer(1, 160, 8, 6, 8, 2, 160, "f32", "gauss_outlier", "gauss_chan", 8, 23, 0),
    Layer(1, 256, 8, 14, 16, 6, 256, "f16", "silu_outlier", "kaiming", 8, 24, 0),
], ids=lambda L: L.name)
def test_codes_and_outputs(layer, shift):
    import torch
    x, w, sB, sG = wl.make_tensors(layer)
    x[0, 0] = np.round(8 * x[0, 0]) / 8                         # coarse values
    conv, _ = make_conv(layer, (x, w, sB, sG))
    store = torch.zeros(x.size + shift, dtype=torch.float16 if layer.dtype == "f16" else torch.float32, device="cuda")
    xd = store[shift:].view(x.shape)
    xd.copy_(torch.from_numpy(x))
    ref = fq.wfq_full(x, w, layer.m, layer.gs, sB, sG, quant_input=True, quant_output=False)
    for mode, y_scale in ((b.WFQ_Y_TILE, "tile"), (b.WFQ_Y_ROW, "row")):
        b.wfq_plan_set_full_quant(conv.plan, 1, mode)
        y = conv.forward(xd).cpu().numpy()
        conv.check_status()
        assert np.array_equal(conv.buffer(b.WFQ_BUF_XQ).cpu().numpy(), ref.Xq)
        assert np.array_equal(conv.buffer(b.WFQ_BUF_SX).cpu().numpy()[:, :, :conv.T], ref.sX.transpose(0, 2, 1))
        # the output transform of the oracle on the GPU's own Y: equal up to the last rounding to fp32
        Y = conv.buffer(b.WFQ_BUF_Y).cpu().numpy()[:, :, :conv.T].astype(np.float64).transpose(0, 2, 1)
        tiles, _ = fq.output_transform_int(Y, ref.AT, y_scale)
        want = orc.scatter_tiles(tiles, layer.N, layer.H, layer.W, layer.m)
        assert np.max(np.abs(y - want)) <= 2.0 ** -23 * np.max(np.abs(want))
    conv.close()


def _check(conv, layer, xd, ref, rows=("tile", "row")):
    """Codes and scales bit for bit, outputs continued from the GPU's own Y, and the epilogue on them."""
    import torch
    bias = torch.linspace(-1, 1, layer.K, device="cuda")
    for y_scale in rows:
        b.wfq_plan_set_full_quant(conv.plan, 1, b.WFQ_Y_TILE if y_scale == "tile" else b.WFQ_Y_ROW)
        conv.set_epilogue(None, b.WFQ_ACT_NONE)
        yd = conv.forward(xd)
        conv.check_status()
        assert np.array_equal(conv.buffer(b.WFQ_BUF_XQ).cpu().numpy(), ref.Xq)
        assert np.array_equal(conv.buffer(b.WFQ_BUF_SX).cpu().numpy()[:, :, :conv.T], ref.sX.transpose(0, 2, 1))
        Y = conv.buffer(b.WFQ_BUF_Y).cpu().numpy()[:, :, :conv.T].astype(np.float64).transpose(0, 2, 1)
        tiles, _ = fq.output_transform_int(Y, ref.AT, y_scale)
        want = orc.scatter_tiles(tiles, layer.N, layer.H, layer.W, layer.m)
        assert np.max(np.abs(yd.cpu().numpy() - want)) <= 2.0 ** -23 * np.max(np.abs(want))
        conv.set_epilogue(bias, b.WFQ_ACT_RELU)
        assert torch.equal(conv.forward(xd), torch.relu(yd + bias[None, :, None, None]))


# More work items than the device holds CTAs (at most four per SM, 592), so that CTAs take a second item: two
# strip buffers (pairs; 16-byte pieces), then one (16-byte pieces; fp32 and groups of 256, one CTA per SM)
@pytest.mark.parametrize("layer", [
    Layer(12, 64, 8, 52, 52, 4, 32, "f16", "silu_outlier", "kaiming", 8, 50, 0),      # 780 items
    Layer(26, 64, 8, 24, 24, 2, 64, "f16", "silu_outlier", "kaiming", 8, 51, 0),      # 624
    Layer(9, 128, 8, 60, 48, 6, 64, "f16", "relu_heavy", "kaiming", 8, 52, 0),        # 720, three CTAs per SM
    Layer(3, 256, 8, 53, 54, 6, 256, "f32", "gauss_outlier", "kaiming", 8, 53, 0),    # 243
], ids=lambda L: L.name)
def test_ctas_with_several_items(layer):
    import torch
    x, w, sB, sG = wl.make_tensors(layer)
    conv, _ = make_conv(layer, (x, w, sB, sG))
    ref = fq.wfq_full(x, w, layer.m, layer.gs, sB, sG, quant_input=True, quant_output=False)
    _check(conv, layer, torch.from_numpy(x).cuda(), ref)
    conv.close()


# Output stores: whole-pair, single-element and 16-byte variants; for F(6,3) CTAs of 64 and of 128 tiles, a second
# CTA along the tiles, and its first and last thread
@pytest.mark.parametrize("m,N,H,W", [
    (6, 13, 30, 5), (6, 13, 30, 6), (6, 43, 17, 5), (6, 43, 17, 6), (6, 50, 30, 5), (6, 50, 30, 6), (6, 2, 66, 65),
    (6, 2, 66, 66), (4, 3, 20, 14), (4, 33, 7, 6), (4, 3, 20, 9), (4, 3, 44, 8), (2, 3, 10, 9), (2, 9, 10, 10)],
    ids=lambda v: str(v))
def test_output_stores(m, N, H, W):
    import torch
    layer = Layer(N, 32, 5, H, W, m, 32, "f16", "silu_outlier", "kaiming_chan", 8, 60, W)
    x, w, sB, sG = wl.make_tensors(layer)
    conv, _ = make_conv(layer, (x, w, sB, sG))
    ref = fq.wfq_full(x, w, m, layer.gs, sB, sG, quant_input=True, quant_output=False)
    _check(conv, layer, torch.from_numpy(x).cuda(), ref)
    conv.close()


def _near_ties(rng, shape, dtype):
    """Odd multiples of 1/16, a third of them moved to a neighbouring float: with an abs-max of 127/8 the scale is
    1/8 exactly and the quotients are half-integers or next to them."""
    v = ((2 * rng.integers(0, 127, shape) + 1) / 16 * rng.choice([-1.0, 1.0], shape)).astype(dtype)
    step = rng.integers(0, 3, shape)
    return np.where(step == 1, np.nextafter(v, dtype(100)), np.where(step == 2, np.nextafter(v, dtype(-100)), v)).astype(dtype)


@pytest.mark.parametrize("m,gs,dtype", [(2, 32, "f32"), (4, 64, "f16"), (4, 96, "f32"), (6, 32, "f16"), (6, 128, "f32")],
                         ids=lambda v: str(v))
def test_input_codes_at_ties(m, gs, dtype):
    import torch
    layer = Layer(2, 2 * gs, 8, 17, 16, m, gs, dtype, "gauss", "kaiming", 8, 70, m)
    _, w, sB, sG = wl.make_tensors(layer)
    rng = np.random.default_rng(m)
    x = _near_ties(rng, (layer.N, layer.C, layer.H, layer.W), np.float16 if dtype == "f16" else np.float32)
    x[:, ::gs, ::m, ::m] = 127 / 8                                # the first pixel of every tile, one channel per group
    ref = fq.wfq_full(x, w, m, gs, sB, sG, quant_input=True, quant_output=False)
    assert np.all(ref.inp.sqx == 0.125)
    q = fq.gather_patches(x, m) * 8
    tie = np.abs(q - np.trunc(q)) == 0.5
    up = np.rint(np.where(tie, q, 0.0)) > np.where(tie, q, 0.0)
    near = ~tie & (np.abs(np.abs(q - np.trunc(q)) - 0.5) < 1e-4)
    assert (tie & up).sum() > 1000 and (tie & ~up).sum() > 1000 and (dtype == "f16" or near.sum() > 1000)
    conv, _ = make_conv(layer, (x, w, sB, sG))
    _check(conv, layer, torch.from_numpy(x).cuda(), ref, rows=("tile",))
    conv.close()


@pytest.mark.parametrize("y_scale", ["tile", "row"])
@pytest.mark.parametrize("m", [2, 4, 6])
def test_output_codes_at_ties(m, y_scale):
    import torch
    layer = Layer(2, 32, 8, 17, 16, m, 32, "f32", "gauss", "kaiming", 8, 71, m)
    conv, (x, w, sB, sG) = make_conv(layer)
    rng = np.random.default_rng(m)
    Y = _near_ties(rng, (conv.P, layer.K, conv.Tp), np.float32)
    n = m + 2
    rows = np.arange(n)
    Y[rows * n + rows % n] = 127 / 8                             # one per row of the n x n matrix
    conv.write_buffer(b.WFQ_BUF_Y, torch.from_numpy(Y))
    mats = orc.matrices(m, sB, sG, None)
    tiles, parts = fq.output_transform_int(Y[:, :, :conv.T].astype(np.float64).transpose(0, 2, 1),
                                           mats.VA * mats.sA[None, :], y_scale)
    assert np.all(parts.sqY == 0.125)
    want = orc.scatter_tiles(tiles, layer.N, layer.H, layer.W, m)
    b.wfq_plan_set_full_quant(conv.plan, 0, b.WFQ_Y_TILE if y_scale == "tile" else b.WFQ_Y_ROW)
    y = torch.full((layer.N, layer.K, layer.H, layer.W), float("nan"), device="cuda")
    b.wfq_output_transform(conv.plan, y.data_ptr(), conv._stream())
    got = y.cpu().numpy()
    assert np.max(np.abs(got - want)) <= 2.0 ** -23 * np.max(np.abs(want))
    conv.close()
