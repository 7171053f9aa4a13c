"""Offline filter path at the edges of its kernel: runs of 128 channels that end early, groups of one to
eight runs of 32 channels, a last block of fewer than eight output channels, filters that are only
4-byte aligned, outputs that are only 1-byte aligned, and groups that hold NaN or infinities."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2412_19867_b200 import binding as b
from tests.gpu_util import codes_close, scales_close

pytestmark = pytest.mark.gpu


def _prepare(w, m, gs, bits=8, shift=0):
    """(codes [P][K][C], scales [P][G][K]) of the plan and, at 8 bits, of the allocation-free call."""
    import torch
    K, C = w.shape[:2]
    store = torch.zeros(w.size + shift, dtype=torch.float32, device="cuda")
    wd = store[shift:].view(w.shape)
    wd.copy_(torch.from_numpy(w))
    conv = b.Conv(1, C, K, 8, 8, m, gs, "f16")
    conv.set_weight_bits(bits)
    conv.prepare(wd)
    q = conv.buffer(b.WFQ_BUF_WQ).cpu().numpy()
    s = conv.buffer(b.WFQ_BUF_SW).cpu().numpy()
    assert not s[:, :, K:].any()
    s = s[:, :, :K]
    if bits == 8:
        codes = torch.full((q.size + shift,), 99, dtype=torch.int8, device="cuda")[shift:]
        scales = torch.full((s.size,), float("nan"), dtype=torch.float32, device="cuda")
        b.wfq_quantize_filters_static(wd.data_ptr(), K, C, m, gs, None, codes.data_ptr(), scales.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream)
        assert np.array_equal(codes.cpu().numpy(), q.ravel())
        assert np.array_equal(scales.cpu().numpy().view(np.int32), s.ravel().view(np.int32))
    conv.close()
    return q, s


@pytest.mark.parametrize("m", [2, 4, 6])
@pytest.mark.parametrize("gs,C,K,bits,shift", [
    (32, 32, 1, 8, 0), (32, 160, 9, 8, 1), (64, 64, 8, 8, 0), (64, 192, 17, 4, 0), (96, 192, 7, 8, 1),
    (128, 384, 8, 8, 0), (160, 160, 9, 4, 0), (224, 448, 5, 8, 0), (256, 256, 15, 8, 1)])
def test_filter_path_matches_oracle(m, gs, C, K, bits, shift):
    rng = np.random.default_rng(1000 * m + C + K)
    w = (rng.standard_normal((K, C, 3, 3)) * np.exp(2 * rng.standard_normal((K, 1, 1, 1)))).astype(np.float32)
    w[0, :gs] = 0.0                                            # a group of zeros: scale 0, codes 0
    q, s = _prepare(w, m, gs, bits, shift)
    ref = orc.prepare_filters(w, m, gs, orc.matrices(m), bits=bits)
    codes_close(q, ref.Wq)
    scales_close(s, ref.sW.transpose(0, 2, 1), rtol=1e-6)


@pytest.mark.parametrize("m", [2, 4, 6])
def test_non_finite_filters_stay_in_their_group(m):
    """The group abs-max ignores NaN, an infinite scale gives codes 0, other groups are unaffected."""
    rng = np.random.default_rng(m)
    K, C, gs = 9, 192, 64
    w = rng.standard_normal((K, C, 3, 3)).astype(np.float32)
    bad = w.copy()
    bad[2, 5] = np.nan
    bad[3, 70] = np.inf
    bad[8, 130, 1, 1] = 3e38                                   # overflows fp32 in some positions
    q0, s0 = _prepare(w, m, gs)
    q, s = _prepare(bad, m, gs)
    hit = np.zeros((K, C // gs), dtype=bool)
    hit[2, 0] = hit[3, 1] = hit[8, 2] = True
    for k in range(K):
        for g in range(C // gs):
            part = slice(g * gs, (g + 1) * gs)
            if not hit[k, g]:
                assert np.array_equal(q[:, k, part], q0[:, k, part]) and np.array_equal(s[:, g, k], s0[:, g, k])
    assert not q[:, 2, 5].any()                                # NaN: code 0
    others = np.delete(np.arange(gs), 5)
    assert np.isfinite(s[:, 0, 2]).all() and q[:, 2, others].any()
    assert not q[:, 3, 64:128][~np.isfinite(s[:, 1, 3])].any()  # scale infinite: codes 0
