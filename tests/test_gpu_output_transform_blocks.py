"""The F(6,3) output transform around its two CTA sizes (64 and 128 tiles): every level against the oracle
for tile counts at the edges of both, with whole-pair and single-element stores, and the epilogue variant
against the plain one."""
import pytest

from paper_2412_19867_b200 import binding as b
from paper_2412_19867_b200.workloads import Layer
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W", [(1, 6, 6), (1, 6, 5), (16, 12, 12), (13, 30, 5), (43, 17, 6), (8, 24, 36), (43, 18, 7)],
                         ids=lambda v: str(v))          # 1, 1, 64, 65, 129, 192, 258 tiles
def test_tile_counts(N, H, W):
    import torch
    layer = Layer(N, 64, 24, H, W, 6, 64, "f16", "relu_heavy", "kaiming", 8, 40, N % 7)
    gu.check_layer_all_levels(layer)
    conv, (x, _, _, _) = gu.make_conv(layer)
    xd = torch.from_numpy(x).cuda()
    plain = conv.forward(xd)
    bias = torch.linspace(-2, 2, layer.K, device="cuda")
    conv.set_epilogue(bias, b.WFQ_ACT_RELU)
    want = torch.relu(plain + bias[None, :, None, None])
    assert torch.equal(conv.forward(xd), want)
    conv.set_output_dtype("f16")
    assert torch.equal(conv.forward(xd), want.half())
    conv.check_status()
    conv.close()
