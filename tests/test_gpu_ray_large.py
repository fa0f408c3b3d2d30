"""The ray kernels that only larger images or batches reach (152 SMs), against the FP64
oracle within the tolerances of test_gpu_ray_batch.py, and image by image, bit by bit.

Forward, one or two images per CTA: one angle per CTA (few CTAs) and two, staged rows of
one batch of loads, of parts of one and of several (300 bins over 600 pixels)."""

import numpy as np
import pytest

from oracle import ray as R

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _randn(*shape):
    return torch.randn(shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(sum(shape)))


@pytest.mark.parametrize("n,A,D,B", [(600, 5, 849, 1), (600, 4, 849, 2), (600, 4, 300, 1), (545, 3, 100, 2),
                                     (130, 90, 184, 4), (130, 90, 184, 14)])
def test_forward(n, A, D, B):
    from paper_2006_04591_gb300.ray import RayTransform
    op = RayTransform(n, A, D, device=0)
    x = _randn(B, n, n)
    p = op.forward(x)
    want = R.forward(x.cpu().numpy(), A, D)
    for b in range(B):
        tol = 1e-6 * n * x[b].abs().max().item() + 1e-6 * np.abs(want[b]).max()
        assert np.abs(p[b].cpu().numpy() - want[b]).max() <= tol
        assert torch.equal(op.forward(x[b:b + 1])[0], p[b])


# Adjoint: tiles of staged bins with one and two images per CTA (600 x 600; 545 is the
# smallest), and the untiled kernel with two pixels per thread and one, two and four
# images (400 x 400; 9001 bins are too narrow for a staging).
@pytest.mark.parametrize("n,A,D,B", [(600, 5, 849, 1), (600, 5, 849, 2), (600, 4, 849, 3), (545, 3, 400, 1),
                                     (400, 4, 566, 1), (400, 4, 566, 2), (400, 3, 566, 4), (600, 3, 9001, 1)])
def test_adjoint(n, A, D, B):
    from paper_2006_04591_gb300.ray import RayTransform
    op = RayTransform(n, A, D, device=0)
    y = _randn(B, A, D)
    g = op.adjoint(y)
    want = R.adjoint(y.cpu().numpy(), n)
    bins = 3 * max(1.0, D / (np.sqrt(2) * n))           # bins whose rays touch a pixel
    for b in range(B):
        tol = 1e-6 * n * y[b].abs().max().item() * (2.9 / n) * bins * A + 1e-6 * np.abs(want[b]).max()
        assert np.abs(g[b].cpu().numpy() - want[b]).max() <= tol
        assert torch.equal(op.adjoint(y[b:b + 1])[0], g[b])
