"""The fully quantized mode switched on at every point of a plan's life: before the workspace, after it, after a
forward, with a change of the input type in between, and with host buffers that are cut into chunks.  Launch
shapes and attributes of its input transform are set when the mode is first known, and only then."""
import pytest

from paper_2412_19867_b200 import binding as b

pytestmark = pytest.mark.gpu

N, C, K, H, W, GS = 8, 128, 24, 40, 48, 128


def _tensors(dtype):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((N, C, H, W), generator=gen, device="cuda").half().to(dtype)
    return x, torch.randn((K, C, 3, 3), generator=gen, device="cuda")


def _run(plan, x):
    import torch
    y = torch.full((N, K, H, W), float("nan"), device="cuda")
    b.wfq_conv_forward(plan, x.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert torch.isfinite(y).all()
    return y


@pytest.mark.parametrize("m", [2, 4, 6])
def test_every_order_of_calls_gives_the_same(m):
    import torch
    stream = torch.cuda.current_stream().cuda_stream
    results = {}
    for order in ("before_workspace", "after_workspace", "after_forward", "f32_first", "off_and_on"):
        x, w = _tensors(torch.float16)
        plan = b.wfq_plan_create(N, C, K, H, W, m, 3, GS, 8)
        b.wfq_plan_set_input_dtype(plan, b.WFQ_F32 if order == "f32_first" else b.WFQ_F16)
        if order == "before_workspace":
            b.wfq_plan_set_full_quant(plan, 1, b.WFQ_Y_TILE)
        nbytes = b.wfq_plan_workspace_bytes(plan)
        ws = torch.empty(nbytes + 1024, dtype=torch.uint8, device="cuda")
        b.wfq_plan_set_workspace(plan, (ws.data_ptr() + 1023) // 1024 * 1024, nbytes)
        if order in ("after_workspace", "f32_first", "off_and_on"):
            b.wfq_plan_set_full_quant(plan, 1, b.WFQ_Y_TILE)
        b.wfq_prepare_filters(plan, w.data_ptr(), stream=stream)
        if order == "after_forward":
            plain = _run(plan, x)
            b.wfq_plan_set_full_quant(plan, 1, b.WFQ_Y_TILE)
        if order == "f32_first":
            results["f32"] = _run(plan, x.float())
            b.wfq_plan_set_input_dtype(plan, b.WFQ_F16)
        if order == "off_and_on":
            b.wfq_plan_set_full_quant(plan, 0, b.WFQ_Y_FP32)
            again = _run(plan, x)
            b.wfq_plan_set_full_quant(plan, 1, b.WFQ_Y_TILE)
        results[order] = _run(plan, x)
        b.wfq_plan_destroy(plan)
    first = results["before_workspace"]
    assert all(torch.equal(first, r) for r in results.values())      # fp16 values in fp32 give the same codes
    assert torch.equal(plain, again) and not torch.equal(plain, first)


def test_chunked_host_buffers():
    import torch
    n, c, h = 12, 64, 96                                              # 14 MB in, 57 MB out: four chunks
    gen = torch.Generator(device="cuda").manual_seed(4)
    x = torch.randn((n, c, h, h), generator=gen, device="cuda").half()
    w = torch.randn((128, c, 3, 3), generator=gen, device="cuda")
    xh = torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)
    yh = torch.empty((n, 128, h, h), dtype=torch.float32, pin_memory=True)
    conv = b.Conv(n, c, 128, h, h, 4, 64, "f16")
    conv.prepare(w)
    for quant in (0, 1, 0, 1):                                        # the chunk plans exist from the first call on
        b.wfq_plan_set_full_quant(conv.plan, quant, b.WFQ_Y_ROW if quant else b.WFQ_Y_FP32)
        yh.fill_(float("nan"))
        conv.forward_host(xh, yh)
        assert torch.equal(yh, conv.forward(x).cpu()), quant
    conv.check_status()
    conv.close()
    conv = b.Conv(n, c, 128, h, h, 4, 64, "f16")
    conv.prepare(w)
    b.wfq_plan_set_full_quant(conv.plan, 1, b.WFQ_Y_ROW)              # before the chunk plans exist
    last = yh.clone()
    conv.forward_host(xh, yh)
    assert torch.equal(yh, last)
    conv.close()
