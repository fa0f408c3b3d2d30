"""The ray kernels share one CTA's positions and weights between one, two or
four images, chosen by the batch; every choice has to give each image what it
gets alone (the same float32 operations in the same order: equal bits), and
that has to match the FP64 oracle within the tolerance of test_gpu_ray.py.
Sizes: rows of several staged blocks and ragged ones, fewer and more bins than
a CTA's 256, bins much narrower and much wider than a pixel, angles that pair
up and that do not."""

import numpy as np
import pytest

from oracle import ray as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,A,D,B", [(64, 30, 91, 301), (37, 7, 53, 403), (50, 3, 300, 330),
                                     (96, 45, 64, 130), (16, 8, 2000, 90), (2, 5, 3, 1300),
                                     (130, 16, 520, 25), (33, 90, 47, 61)])
def test_batch_equals_single_images(n, A, D, B):
    from paper_2006_04591_gb300.ray import RayTransform
    op = RayTransform(n, A, D, device=0)
    gen = torch.Generator(device="cuda").manual_seed(n + D)
    x = torch.randn((B, n, n), device="cuda", generator=gen)
    y = torch.randn((B, A, D), device="cuda", generator=gen)
    p, g = op.forward(x), op.adjoint(y)
    some = sorted({0, 1, 2, 3, B // 2, B - 2, B - 1})
    for b in some:
        assert torch.equal(p[b], op.forward(x[b:b + 1])[0]), b
        assert torch.equal(g[b], op.adjoint(y[b:b + 1])[0]), b
    xs, ys = x[some].cpu().numpy(), y[some].cpu().numpy()
    want_p, want_g = R.forward(xs, A, D), R.adjoint(ys, n)
    for k, b in enumerate(some):
        tol = 1e-6 * n * np.abs(xs[k]).max() + 1e-6 * np.abs(want_p[k]).max()
        assert np.abs(p[b].cpu().numpy() - want_p[k]).max() <= tol
        bins = 3 * max(1.0, D / (np.sqrt(2) * n))       # bins whose rays touch a pixel
        tol = 1e-6 * n * np.abs(ys[k]).max() * (2.9 / n) * bins * A + 1e-6 * np.abs(want_g[k]).max()
        assert np.abs(g[b].cpu().numpy() - want_g[k]).max() <= tol


def test_infinite_bin_reaches_only_its_rays_pixels():
    from paper_2006_04591_gb300.ray import RayTransform
    n, A, D = 40, 6, 57
    op = RayTransform(n, A, D, device=0)
    y = torch.zeros((1, A, D), device="cuda")
    y[0, 2, 30] = float("inf")
    hit = torch.isfinite(op.adjoint(y)[0]).logical_not().cpu().numpy()
    e = np.zeros((1, A, D), np.float32)
    e[0, 2, 30] = 1.0
    assert not np.any(hit & (np.abs(R.adjoint(e, n)[0]) < 1e-9))
