"""The weight gradient of layers wider than one tensor-core tile (42 input
channels): groups in one launch, against the float64 gradient of the
bfloat16-rounded operands (1e-4 of the largest, the sums' float32 rounding, as in
test_gpu_nn_tc.py) and, bit by bit, against the groups run one by one."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Ci,Co,H,W", [(1, 43, 32, 3, 128), (2, 84, 16, 5, 64), (1, 85, 5, 4, 182),
                                         (4, 102, 32, 16, 128), (1, 130, 96, 2, 18), (3, 41, 8, 3, 130)])
def test_wide_weight_gradient(B, Ci, Co, H, W):
    from paper_2006_04591_gb300 import nn
    gen = torch.Generator().manual_seed(Ci + W)
    x = torch.randn((B, Ci, H, W), generator=gen)
    gout = torch.randn((B, Co, H, W), generator=gen)
    xc, gc = x.cuda(), gout.cuda()
    gw, gb = torch.empty((Co, Ci, 3, 3), device="cuda"), torch.empty(Co, device="cuda")
    nn.shl_nn_conv3x3_backward_weight_tc_wide(xc, gc, gw, gb)
    nn.shl_nn_tc_status()
    bf = lambda t: t.to(torch.bfloat16).double()  # noqa: E731
    want = torch.nn.grad.conv2d_weight(bf(x), (Co, Ci, 3, 3), bf(gout), padding=1)
    assert (gw.double().cpu() - want).abs().max() <= 1e-4 * want.abs().max()
    wb = gout.double().sum((0, 2, 3))
    assert (gb.double().cpu() - wb).abs().max() <= 1e-5 * wb.abs().max()
    for c0 in range(0, Ci, 42):
        c1 = min(Ci, c0 + 42)
        gg = torch.empty((Co, c1 - c0, 3, 3), device="cuda")
        nn.shl_nn_conv3x3_backward_weight_tc(xc[:, c0:c1].contiguous(), gc, gg, torch.empty_like(gb))
        assert torch.equal(gw[:, c0:c1], gg)


def test_wide_layer_takes_views_that_start_anywhere():
    from paper_2006_04591_gb300 import nn
    g = torch.Generator(device="cuda").manual_seed(1)
    base = torch.randn(1 + 64 * 4 * 32, device="cuda", generator=g)
    x = base[1:].view(1, 64, 4, 32)                      # 4 bytes past a 16-byte boundary
    w = torch.randn((64, 64, 3, 3), device="cuda", generator=g, requires_grad=True)
    b = torch.zeros(64, device="cuda", requires_grad=True)
    gy = torch.randn((1, 64, 4, 32), device="cuda", generator=g)
    gw = torch.autograd.grad(nn.conv3x3(x, w, b, tc=True), w, gy)[0]
    want = torch.autograd.grad(nn.conv3x3(x.clone(), w, b, tc=True), w, gy)[0]
    assert torch.equal(gw, want)
