"""The fully quantized transforms where their staging and stores change form: rows copied in 16-byte
pieces, in pairs or one by one, x that is only 4-byte aligned, group sizes without a register variant,
fp32 input, every store variant of the output transform, and codes at ties."""
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
    x[0, 0] = np.round(8 * x[0, 0]) / 8                         # values that meet ties of their group's scale
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
