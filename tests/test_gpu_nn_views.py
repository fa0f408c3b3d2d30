"""The launch wrappers of the learned parts take any view: a kernel gets addresses of
row-major data, so transposed or strided operands (one or several in a call) are copied
first, each copy living until the launch, and outputs are row-major.  Against the same
call on contiguous copies: equal bits."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _view(t, kind):
    """The values of t behind other strides."""
    if kind == "plain":
        return t
    if kind == "transposed":
        return t.transpose(-1, -2).contiguous().transpose(-1, -2)
    wide = torch.zeros(t.shape[:-1] + (2 * t.shape[-1],), dtype=t.dtype, device=t.device)
    wide[..., ::2] = t
    return wide[..., ::2]


KINDS = ("plain", "transposed", "strided")


@pytest.mark.parametrize("kf", KINDS)
@pytest.mark.parametrize("km", KINDS)
@pytest.mark.parametrize("kx", KINDS)
def test_mask_mix(kf, km, kx):
    from paper_2006_04591_gb300 import nn
    g, shape = _gen(3), (3, 24, 40)
    fm, f, gu = (torch.randn(shape, device="cuda", generator=g) for _ in range(3))
    mask = (torch.rand(shape, device="cuda", generator=g) < 0.5).to(torch.uint8)
    for _ in range(3):                       # the allocator's blocks come back in turn
        leaf = _view(f, kf).detach().requires_grad_(True)
        u = nn.mask_mix(_view(fm, kx), _view(mask, km), leaf)
        (gf,) = torch.autograd.grad(u, (leaf,), _view(gu, kf))
        assert torch.equal(u, torch.where(mask.bool(), fm, f))
        assert torch.equal(gf, torch.where(mask.bool(), torch.zeros_like(gu), gu))


@pytest.mark.parametrize("kx", KINDS)
@pytest.mark.parametrize("kw", KINDS)
@pytest.mark.parametrize("kg", KINDS)
def test_linear(kx, kw, kg):
    from paper_2006_04591_gb300 import nn
    g = _gen(4)
    x, w = torch.randn((6, 32), device="cuda", generator=g), torch.randn((20, 32), device="cuda", generator=g)
    b, gy = torch.randn(20, device="cuda", generator=g), torch.randn((6, 20), device="cuda", generator=g)

    def run(x, w, b, gy):
        x, w, b = (t.detach().requires_grad_(True) for t in (x, w, b))
        y = nn.linear(x, w, b)
        return (y,) + torch.autograd.grad(y, (x, w, b), gy)

    for a, c in zip(run(_view(x, kx), _view(w, kw), _view(b, "plain" if kw == "plain" else "strided"),
                        _view(gy, kg)), run(x, w, b, gy)):
        assert torch.equal(a, c)


@pytest.mark.parametrize("kind", KINDS[1:])
def test_gate_prelu_and_heads(kind):
    from paper_2006_04591_gb300 import nn
    g = _gen(5)
    c, gy = (torch.randn((2, 4, 16, 24), device="cuda", generator=g) for _ in range(2))
    d = torch.rand((2, 4), device="cuda", generator=g) + 0.3
    s = torch.rand(4, device="cuda", generator=g) + 0.5
    a = torch.tensor([0.3], device="cuda")

    def run(v):
        cl, dl = v(c).detach().requires_grad_(True), v(d).detach().requires_grad_(True)
        y = nn.gate(cl, dl, 0.1, scale=s if v is plain else _view(s, "strided"))
        out = [y, *torch.autograd.grad(y, (cl, dl), v(gy))]
        y = nn.prelu(cl, a)
        out += [y, *torch.autograd.grad(y, (cl,), v(gy))]
        y = nn.softplus(nn.gap(cl))
        out += [y, *torch.autograd.grad(y, (cl,), v(d)), nn.avgpool(v(c), 4)]
        t = torch.empty((4, 2, 4), device="cuda")
        out.append(nn.scale_thresholds(v(c[:, :, 0, :4]), s if v is plain else _view(s, "strided"), t))
        return out

    plain = lambda t: t  # noqa: E731
    for got, want in zip(run(lambda t: _view(t, kind)), run(plain)):
        assert torch.equal(got, want)


def test_masks_that_do_not_cover_the_image():
    from paper_2006_04591_gb300 import nn
    f = torch.randn((2, 8, 12), device="cuda")
    mask = torch.ones((2, 8, 12), dtype=torch.uint8, device="cuda")
    for fm, m in ((f, mask[0]), (f[0], mask), (f, mask.float())):
        with pytest.raises(ValueError):
            nn.mask_mix(fm, m, f)
    row = (torch.arange(12, device="cuda") % 2).to(torch.uint8).expand(2, 8, 12)
    assert torch.equal(nn.mask_mix(f, row, -f), torch.where(row.bool(), f, -f))
