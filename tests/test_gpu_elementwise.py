"""The vectorised elementwise kernels of the learned parts at the sizes where
their four-element bodies can go wrong (fewer elements than a body, remainders,
several grid strides, pointers that are not 16-byte aligned), against float64.
Outputs are single roundings of the same expressions (2e-6 of the largest);
sums of n terms in float32 partials are held to 1e-5 of the sum of magnitudes."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _near(a, b, tol=2e-6):
    assert (a.double() - b).abs().max().item() <= tol * max(b.abs().max().item(), 1e-30)


@pytest.mark.parametrize("n", [1, 3, 4, 1021, 4096, 5003, (1 << 21) + 7])
@pytest.mark.parametrize("shift", [0, 1])
def test_prelu_and_mask_mix(n, shift):
    from paper_2006_04591_gb300 import nn
    g = _gen(n + shift)
    x = torch.randn(n + shift, device="cuda", generator=g)[shift:].requires_grad_(True)
    gy = torch.randn(n + shift, device="cuda", generator=g)[shift:]
    a = torch.tensor([0.3], device="cuda", requires_grad=True)
    y = nn.prelu(x, a)
    gx, ga = torch.autograd.grad(y, (x, a), gy)
    xd, gd = x.detach().double(), gy.double()
    _near(y.detach(), torch.where(xd >= 0, xd, a.detach().double() * xd))
    _near(gx, torch.where(xd >= 0, gd, a.detach().double() * gd))
    t = torch.where(xd < 0, gd * xd, torch.zeros_like(xd))
    assert abs(ga.item() - t.sum().item()) <= 1e-5 * t.abs().sum().item() + 1e-12
    m = (torch.rand(n + shift, device="cuda", generator=g) < 0.5).to(torch.uint8)[shift:]
    f = gy.clone().requires_grad_(True)
    u = nn.mask_mix(x.detach(), m, f)
    assert torch.equal(u, torch.where(m.bool(), x.detach(), f.detach()))
    (gf,) = torch.autograd.grad(u, (f,), gy)
    assert torch.equal(gf, torch.where(m.bool(), torch.zeros_like(gy), gy))


@pytest.mark.parametrize("H,W", [(1, 1), (1, 3), (2, 2), (7, 9), (64, 60), (300, 301), (512, 512)])
@pytest.mark.parametrize("scaled", [False, True])
def test_gate(H, W, scaled):
    from paper_2006_04591_gb300 import nn
    B, K, tau = 2, 3, 0.1
    g = _gen(H * 1000 + W)
    c = torch.randn((B, K, H, W), device="cuda", generator=g, requires_grad=True)
    d = (torch.rand((B, K), device="cuda", generator=g) + 0.3).requires_grad_(True)
    s = torch.rand(K, device="cuda", generator=g) + 0.5 if scaled else None
    gy = torch.randn(c.shape, device="cuda", generator=g)
    y = nn.gate(c, d, tau, scale=s)
    gc, gd = torch.autograd.grad(y, (c, d), gy)
    cd, dd = c.detach().double().requires_grad_(True), d.detach().double().requires_grad_(True)
    lim = (dd * s.double() if scaled else dd)[:, :, None, None]
    z = cd * torch.sigmoid((cd.abs() / lim - 1.0) / tau)
    wc, wd = torch.autograd.grad(z, (cd, dd), gy.double())
    # (|c|/delta - 1)/tau carries the rounding of |c|/delta times 1/tau
    _near(y.detach(), z.detach(), 2e-5)
    _near(gc, wc, 2e-4)
    mag = (wc * cd.detach()).abs().sum((2, 3)) / dd.detach() + 1e-12
    assert ((gd.double() - wd).abs() <= 1e-4 * mag).all()
