"""The weight gradient of very wide layers: launches of as many input channels as keep the
partial sums within 2^25 floats share one workspace of that size, whatever the number of
channels.  Bit by bit against the groups of 42 run one by one; a layer of 4100 channels
also through conv3x3, against the float64 gradient of the bfloat16-rounded operands (1e-4
of the largest, as in test_gpu_nn_tc.py)."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 40 x 16 x 16: 160 units, one CTA for each of 152 SMs; 252 channels a launch at Co = 96
@pytest.mark.parametrize("B,Ci,Co,H,W", [(1, 126, 16, 3, 32), (2, 127, 5, 4, 18), (40, 252, 96, 16, 16),
                                         (40, 253, 96, 16, 16), (40, 505, 96, 16, 16), (1, 4100, 8, 2, 16)])
def test_slabs(B, Ci, Co, H, W):
    from paper_2006_04591_gb300 import nn
    g = torch.Generator(device="cuda").manual_seed(Ci)
    x = torch.randn((B, Ci, H, W), device="cuda", generator=g)
    gout = torch.randn((B, Co, H, W), device="cuda", generator=g)
    ws = nn.lib().shl_nn_conv3x3_backward_weight_tc_wide_workspace_floats
    bias_partials = 256 * Co                            # at most one CTA per SM
    assert 0 < ws(B, Ci, Co, H, W) <= (1 << 25) + bias_partials
    gw, gb = torch.empty((Co, Ci, 3, 3), device="cuda"), torch.empty(Co, device="cuda")
    nn.shl_nn_conv3x3_backward_weight_tc_wide(x, gout, gw, gb)
    nn.shl_nn_tc_status()
    for c0 in range(0, Ci, 42):
        c1 = min(Ci, c0 + 42)
        gg, gbg = torch.empty((Co, c1 - c0, 3, 3), device="cuda"), torch.empty_like(gb)
        nn.shl_nn_conv3x3_backward_weight_tc(x[:, c0:c1].contiguous(), gout, gg, gbg)
        assert torch.equal(gw[:, c0:c1], gg) and torch.equal(gb, gbg)


def test_layer_of_4100_channels():
    from paper_2006_04591_gb300 import nn
    g = torch.Generator(device="cuda").manual_seed(0)
    x = torch.randn((1, 4100, 4, 16), device="cuda", generator=g)
    w = torch.randn((8, 4100, 3, 3), device="cuda", generator=g, requires_grad=True)
    b = torch.zeros(8, device="cuda", requires_grad=True)
    gy = torch.randn((1, 8, 4, 16), device="cuda", generator=g)
    gw, gb = torch.autograd.grad(nn.conv3x3(x, w, b, tc=True), (w, b), gy)
    bf = lambda t: t.to(torch.bfloat16).double()  # noqa: E731
    want = torch.nn.grad.conv2d_weight(bf(x), (8, 4100, 3, 3), bf(gy), padding=1)
    assert (gw.double() - want).abs().max() <= 1e-4 * want.abs().max()
    assert (gb.double() - gy.double().sum((0, 2, 3))).abs().max() <= 1e-5 * gy.abs().sum((0, 2, 3)).max()
