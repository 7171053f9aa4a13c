"""Kernels whose waits run out end by themselves with their copies landed and their tensor memory free: the status word
says so, and a fresh plan on the same device computes what the first one did."""
import pytest

from paper_2412_19867_b200 import binding as b

pytestmark = pytest.mark.gpu


def _layer(C=192, gs=64, dtype="f16", layout="nchw"):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(C + gs)
    N, K, H, W = 2, 72, 12, 17                       # 30 tiles: units of 64 and 32 columns are cut in both orientations
    x = torch.randn((N, C, H, W), generator=gen, device="cuda").to(torch.float32 if dtype == "f32" else torch.float16)
    w = torch.randn((K, C, 3, 3), generator=gen, device="cuda")
    if layout == "nhwc":
        x = x.permute(0, 2, 3, 1).contiguous()

    def make():
        conv = b.Conv(N, C, K, H, W, 4, gs, dtype)
        conv.set_input_layout(layout)
        conv.prepare(w)
        return conv
    return make, x


def _check_fresh_plan(make, x, want):
    import torch
    conv = make()
    got = conv.forward(x)
    conv.check_status()
    assert torch.equal(got, want)
    conv.close()


@pytest.mark.parametrize("stage", [0, 1])
@pytest.mark.parametrize("gs", [32, 64, 96])
@pytest.mark.parametrize("shape", [0, 164, 264, 248, 232, 116])
def test_starved_contraction(shape, gs, stage):
    import torch
    make, x = _layer(gs=gs)
    conv = make()
    want = conv.forward(x)
    conv.check_status()
    b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_GEMM_SHAPE, shape)
    b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_WAIT_CYCLES, 2_000_000)      # about 1 ms
    b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_SKIP_GEMM_STAGE, stage)
    conv.forward(x)
    torch.cuda.synchronize()
    status, where = b.wfq_check_device_status(conv.plan, conv._stream())
    assert status == b.WFQ_ERR_TIMEOUT and where in range(1, 7)
    conv.close()
    _check_fresh_plan(make, x, want)


@pytest.mark.parametrize("dtype,layout,kernel", [("f16", "nchw", 1), ("f16", "nchw", 2), ("f16", "nhwc", 0),
                                                 ("f16", "nhwc", 1), ("f32", "nhwc", 0)])
@pytest.mark.parametrize("cycles", [1000, 3000, 10000])
def test_limits_shorter_than_the_copies(dtype, layout, kernel, cycles):
    """Waits that run out while what they wait for is on its way (whether they do is up to the hardware's own time
    limit of a try)."""
    import torch
    make, x = _layer(dtype=dtype, layout=layout)
    conv = make()
    want = conv.forward(x)
    conv.check_status()
    b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_INPUT_TRANSFORM_KERNEL, kernel)
    b.wfq_plan_set_debug_option(conv.plan, b.WFQ_DEBUG_WAIT_CYCLES, cycles)
    for _ in range(20):
        conv.forward(x)
    torch.cuda.synchronize()
    status, _ = b.wfq_check_device_status(conv.plan, conv._stream())
    assert status in (b.WFQ_OK, b.WFQ_ERR_TIMEOUT)
    conv.close()
    _check_fresh_plan(make, x, want)
