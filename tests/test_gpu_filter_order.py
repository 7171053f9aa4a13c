"""Filters replaced and used with nothing in between: the contraction streams filter codes before its
dependency wait, so the input transform in front of it has to hold it back until the filter preparation
has completed.  Every input transform, as stream launches and inside one graph."""
import pytest

from paper_2412_19867_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [False, True], ids=["stream", "graph"])
@pytest.mark.parametrize("m,gs,dtype,layout,quant", [
    (6, 64, "f16", "nchw", 0), (4, 32, "f32", "nchw", 0), (4, 64, "f16", "nchw", 1), (6, 64, "f16", "nhwc", 0),
    (2, 96, "f16", "nhwc", 0)], ids=lambda v: str(v))
def test_forward_right_behind_prepare(m, gs, dtype, layout, quant, graph):
    import torch
    N, C, K, H, W = 1, 576, 640, 14, 14                       # few tiles, many filters
    gen = torch.Generator(device="cuda").manual_seed(m)
    shape = (N, H, W, C) if layout == "nhwc" else (N, C, H, W)
    x = torch.randn(shape, generator=gen, device="cuda").to(torch.float16 if dtype == "f16" else torch.float32)
    conv = b.Conv(N, C, K, H, W, m, gs, dtype)
    conv.set_input_layout(layout)
    if quant:
        b.wfq_plan_set_full_quant(conv.plan, 1, b.WFQ_Y_TILE)
    ws = [torch.randn((K, C, 3, 3), generator=gen, device="cuda") for _ in range(2)]
    want = []
    for w in ws:
        conv.prepare(w)
        torch.cuda.synchronize()
        want.append(conv.forward(x))
        torch.cuda.synchronize()
    assert not torch.equal(want[0], want[1])
    ys = [torch.empty_like(want[0]) for _ in range(8)]

    def alternate():
        for i, y in enumerate(ys):
            conv.prepare(ws[i % 2])
            conv.forward(x, y)

    if graph:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            alternate()
        g.replay()
    else:
        alternate()
    torch.cuda.synchronize()
    conv.check_status()
    for i, y in enumerate(ys):
        assert torch.equal(y, want[i % 2]), i
    conv.close()
