"""More planes than a launch can index by blockIdx.y (65535): the transforms split them
over several launches.  Small images in great number, whose subbands all fit the staging
area: the fused shrink equals the decomposition followed by the thresholded
reconstruction, and an image in the last launch equals the same image alone (1e-5 of the
largest value, the float32 tolerance of test_gpu_general.py; the number of subband groups
may depend on the batch)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# one-stage and two-stage lengths as rows and as columns, and a power-of-two plane
@pytest.mark.parametrize("rows,cols,K,B", [(6, 6, 3, 25000), (80, 1, 3, 22000), (1, 80, 2, 33000),
                                           (6, 6, 1, 66000), (16, 16, 1, 66000)])
def test_more_than_65535_planes(rows, cols, K, B):
    from paper_2006_04591_gb300.shearlet import Bank
    rng = np.random.default_rng(rows + K)
    g = rng.random((K, rows, cols)) + 0.5
    bank = Bank.from_spectra(0.5 * (g + np.roll(g[:, ::-1, ::-1], (1, 1), (1, 2))), device=0)
    gen = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((B, rows, cols), device="cuda", generator=gen)
    th = torch.full((B, K), 0.1, device="cuda")
    c = bank.decompose(x)
    y = bank.reconstruct(c)
    tol = 1e-5 * x.abs().max()
    assert (y - x).abs().max() <= 4 * tol               # there and back, as in test_gpu_general.py
    z = bank.reconstruct(c, thresh=th)
    s = bank.shrink(x, th)
    assert (s - z).abs().max() <= tol
    for b in (0, 21844, B - 1):
        one = x[b:b + 1].contiguous()
        assert (bank.decompose(one)[0] - c[b]).abs().max() <= tol
        assert (bank.shrink(one, th[:1])[0] - s[b]).abs().max() <= tol
