"""Edges of the contraction's units.  Output channel counts around the blocks of 64 columns: the first K channels of a
wider layer give the same values bit for bit, and nothing is written beyond them."""
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


@pytest.mark.parametrize("T", [1, 31, 32, 33, 96, 127, 128, 129, 161, 257])
def test_partial_row_blocks(T):
    """Tile counts around the 32 tiles of a store and the 128 of a unit, rows = tiles (stored by TMA) and rows = channels
    (stored by the lanes): within the rounding of the fp32 sums of the scaled group sums in 64 bits, and rows = tiles
    writes nothing behind the 16 bytes of the last tile (the unit of a TMA store; rows of Y are padded to 32 tiles)."""
    import torch
    m, C, K, gs = 4, 192, 72, 64
    gen = torch.Generator(device="cuda").manual_seed(T)
    x = torch.randn((1, C, m, m * T), generator=gen, device="cuda").half()
    conv = b.Conv(1, C, K, m, m * T, m, gs, "f16")
    conv.prepare(torch.randn((K, C, 3, 3), generator=gen, device="cuda"))
    assert conv.T == T
    b.wfq_input_transform_quantize(conv.plan, x.data_ptr(), conv._stream())
    xq, wq = conv.buffer(b.WFQ_BUF_XQ).double(), conv.buffer(b.WFQ_BUF_WQ).double()
    sx, sw = conv.buffer(b.WFQ_BUF_SX).double(), conv.buffer(b.WFQ_BUF_SW).double()
    terms = torch.stack([wq[:, :, g * gs:(g + 1) * gs] @ xq[:, :, g * gs:(g + 1) * gs].transpose(1, 2) *
                         sw[:, g, :K, None] * sx[:, g, None, :T] for g in range(C // gs)])
    # a product with each scale and a sum: each rounds once per group
    bound = (C // gs + 2) * 2.0 ** -24 * terms.abs().sum(0)
    for shape in (264, 248, 232, 164, 116):      # which units are cut is up to the number of SMs: test_cut_units
        b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_GEMM_SHAPE, shape)
        Y = conv.buffer(b.WFQ_BUF_Y).fill_(float("nan"))
        b.wfq_gemm_dequantize(conv.plan, conv._stream())
        assert ((Y[:, :, :T].double() - terms.sum(0)).abs() <= bound).all(), shape
        assert shape >= 200 or torch.isnan(Y[:, :, (T + 3) // 4 * 4:]).all()
    conv.check_status()
    conv.close()


@pytest.mark.parametrize("T,K", [(161, 200), (257, 72), (129, 129), (97, 264)])
@pytest.mark.parametrize("shape,parts", [(164, 2), (264, 2), (248, 3), (232, 2)])
def test_cut_units(shape, parts, T, K):
    """Whole rounds of units followed by a round that is cut into parts of their columns, with ragged tiles and channels:
    equal bit for bit to the same layer on one CTA, where nothing is cut, and nothing else of Y is written.  The CTAs are
    given, so the coverage does not depend on the device: a last round of r units is cut if r * parts of them have
    room, a unit has several chunks (here three groups of 64 channels, two to a chunk) and more columns than a part."""
    import torch
    m, C, gs = 4, 192, 64
    gen = torch.Generator(device="cuda").manual_seed(T + K)
    x = torch.randn((1, C, m, m * T), generator=gen, device="cuda").half()
    conv = b.Conv(1, C, K, m, m * T, m, gs, "f16")
    conv.prepare(torch.randn((K, C, 3, 3), generator=gen, device="cuda"))
    b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_GEMM_SHAPE, shape)
    b.wfq_input_transform_quantize(conv.plan, x.data_ptr(), conv._stream())
    rows, cols, bn = (K, T, shape - 200) if shape >= 200 else (T, K, shape - 100)
    units = conv.P * -(-rows // 128) * -(-cols // bn)

    def contract(ctas):
        b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_GEMM_CTAS, ctas)
        Y = conv.buffer(b.WFQ_BUF_Y).fill_(float("nan"))
        b.wfq_gemm_dequantize(conv.plan, conv._stream())
        conv.check_status()
        return Y.clone()

    want = contract(1)
    assert not torch.isnan(want[:, :, :T]).any()
    cut = [c for c in range(2, units) if 0 < units % c and units % c * parts <= c]
    for ctas in [cut[0], cut[len(cut) // 2], cut[-1], parts * units, 0]:        # several rounds, one, none in front; as chosen
        got = contract(ctas)
        assert torch.equal(got[:, :, :T], want[:, :, :T]), ctas
        assert shape >= 200 or torch.isnan(got[:, :, (T + 3) // 4 * 4:]).all()
    conv.close()
