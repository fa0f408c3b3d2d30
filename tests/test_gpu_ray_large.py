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
