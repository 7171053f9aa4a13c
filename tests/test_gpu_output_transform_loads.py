"""The output transform on both sides of the sizes of Y (32 MiB, and 256 MiB for F(6,3)) at which its loads of
Y change, every store variant and both epilogue variants, against the transform in 64 bits.

Bound: row sums of |A^T| are at most 67 (F(6,3)), so an output is off by at most 6 roundings of 2^-24 each on
67^2 max|Y S_A S_A| (5 for these Y) = 8e-3; the largest outputs are above 4000.  1e-5 of the largest output
leaves a factor of five.
"""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2412_19867_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,N,H,W,K", [
    (6, 4, 48, 48, 511), (6, 4, 48, 48, 512),              # 256 tiles: 32 MiB at 512 channels
    (6, 1, 81, 81, 585), (6, 1, 81, 81, 586),              # 196 tiles, odd W, CTAs of 64 tiles
    (6, 8, 96, 96, 512), (6, 8, 96, 96, 513),              # 2048 tiles: 256 MiB at 512 channels
    (4, 2, 64, 64, 455), (4, 2, 64, 64, 456), (4, 2, 62, 62, 456), (4, 2, 61, 61, 456),
    (2, 2, 64, 64, 255), (2, 2, 64, 64, 256), (2, 2, 63, 63, 256)], ids=lambda v: str(v))
def test_sizes_of_y(m, N, H, W, K):
    import torch
    conv = b.Conv(N, 32, K, H, W, m, 32, "f16")
    gen = torch.Generator(device="cuda").manual_seed(K)
    conv.prepare(torch.zeros((K, 32, 3, 3), device="cuda"))
    Y = conv.buffer(b.WFQ_BUF_Y)
    mats = orc.matrices(m)
    n, TH, TW = m + 2, -(-H // m), -(-W // m)
    Y.copy_(torch.randn(Y.shape, generator=gen, device="cuda"))
    Y.div_(torch.tensor(np.outer(mats.sA, mats.sA).reshape(-1, 1, 1), dtype=torch.float32, device="cuda"))
    AT = torch.tensor(mats.VA * mats.sA[None, :], dtype=torch.float64, device="cuda")
    ks = torch.tensor(sorted({0, 1, K // 2, K - 1}), device="cuda")
    tiles = Y[:, ks, :conv.T].double().reshape(n, n, len(ks), N, TH, TW)
    want = torch.einsum("ui,ijkbhw,vj->bkhuwv", AT, tiles, AT).reshape(N, len(ks), TH * m, TW * m)[:, :, :H, :W]
    y = torch.full((N, K, H, W), float("nan"), device="cuda")
    b.wfq_output_transform(conv.plan, y.data_ptr(), conv._stream())
    assert torch.isfinite(y).all()
    assert float((y[:, ks].double() - want).abs().max()) <= 1e-5 * float(want.abs().max())
    bias = torch.linspace(-2, 2, K, device="cuda")
    conv.set_epilogue(bias, b.WFQ_ACT_RELU)
    y2 = torch.full_like(y, float("nan"))
    b.wfq_output_transform(conv.plan, y2.data_ptr(), conv._stream())
    assert torch.equal(y2, torch.relu(y + bias[None, :, None, None]))
    conv.close()
