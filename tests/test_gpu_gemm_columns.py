"""Output channel counts around the blocks of 64 columns of the contraction and the groups of eight in which a
partial block is stored: the first K channels of a wider layer give the same values bit for bit, and nothing is
written beyond them."""
import pytest

from paper_2412_19867_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bn", [64, 16])
@pytest.mark.parametrize("m,gs", [(4, 32), (6, 64), (2, 128)])
def test_partial_column_blocks(m, gs, bn):
    import torch
    N, C, H, W, full = 2, 128, 26, 23, 192
    gen = torch.Generator(device="cuda").manual_seed(m)
    x = torch.randn((N, C, H, W), generator=gen, device="cuda").half()
    w = torch.randn((full, C, 3, 3), generator=gen, device="cuda")
    want = None
    for K in (full, 1, 2, 7, 8, 9, 16, 17, 55, 63, 64, 65, 71, 72, 73, 127, 129, 191):
        conv = b.Conv(N, C, K, H, W, m, gs, "f16")
        conv.prepare(w[:K].contiguous())
        b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_GEMM_SHAPE, 100 + bn)
        conv.buffer(b.WFQ_BUF_Y).fill_(float("nan"))
        b.wfq_input_transform_quantize(conv.plan, x.data_ptr(), conv._stream())
        b.wfq_gemm_dequantize(conv.plan, conv._stream())
        Y = conv.buffer(b.WFQ_BUF_Y)
        assert not torch.isnan(Y[:, :, :conv.T]).any() and torch.isnan(Y[:, :, conv.T:]).all(), K
        if want is None:
            want = Y[:, :, :conv.T].clone()
        assert torch.equal(Y[:, :, :conv.T], want[:, :K]), K
        conv.check_status()
        conv.close()
