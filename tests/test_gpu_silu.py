"""SiLU of the output transform over the whole range of fp32: the outputs of an all-zero image are the activation of
the bias."""
import pytest

from paper_2412_19867_b200 import binding as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,W", [(4, 8), (6, 7), (2, 6)])
def test_silu_over_the_whole_range(m, W):
    import torch
    t = torch.cat([torch.linspace(-110, 110, 977), torch.logspace(-40, 38, 400), -torch.logspace(-40, 38, 400),
                   torch.tensor([0.0, -0.0, float("inf"), float("-inf"), float("nan")])]).float().cuda()
    conv = b.Conv(1, 32, t.numel(), 6, W, m, 32, "f16")
    conv.prepare(torch.zeros((t.numel(), 32, 3, 3), device="cuda"))
    conv.set_epilogue(t, b.WFQ_ACT_SILU)
    y = conv.forward(torch.zeros((1, 32, 6, W), device="cuda").half())[0]
    assert torch.equal(y.nan_to_num(1.5), y[:, :1, :1].nan_to_num(1.5).expand_as(y))
    got, x = y[:-2, 0, 0].double(), t[:-2].double()
    # exp of the fast kind: 2 + 1.173 |t| units in the last place; sum, reciprocal and product: half a unit each.  Below
    # -88.7 the exponential overflows and the result is 0 instead of less than 3e-37.
    bound = (4 + 1.173 * x.abs()) * 2.0 ** -23 * (x / (1 + torch.exp(-x))).abs() + 3e-37
    want = torch.where(torch.isinf(x), x, x / (1 + torch.exp(-x)))
    finite = ~torch.isinf(x)
    assert ((got - want).abs()[finite] <= bound[finite]).all()
    assert got[-1] == float("inf") and torch.isnan(y[-1]).all() and torch.isnan(y[-2]).all()     # inf; -inf * 0, NaN
    conv.close()
