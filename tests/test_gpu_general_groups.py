"""The column pass that adds the subband groups' partial sums (csrc/general_pairs.cuh)
loads the groups four at a time: subband counts that leave remainders of four, single
groups and more subbands than groups, at direct and Bluestein lengths.  Error measure
and tolerance as in test_gpu_general.py: max |gpu - oracle| / max |oracle| <= 1e-5."""

import numpy as np
import pytest

from oracle import transform as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 3, 4, 5, 7, 8, 15, 16, 17])
@pytest.mark.parametrize("rows", [80, 100, 253, 480])
def test_group_sums(rows, K):
    from paper_2006_04591_gb300.shearlet import Bank
    rng = np.random.default_rng(rows + K)
    cols, B = 9, 2
    g = rng.standard_normal((K - 1, rows, cols))
    g = 0.5 * (g + np.roll(g[:, ::-1, ::-1], (1, 1), (1, 2)))
    G = np.fft.fft2(g, axes=(-2, -1)).real / np.sqrt(rows * cols)
    Wp = np.sum(G ** 2, axis=0)
    G = np.concatenate([G, np.sqrt(1.1 * Wp.max() - Wp)[None]])      # makes W constant
    bank = Bank.from_spectra(G, device=0)
    assert bank.general and bank.K == K
    c = rng.standard_normal((B, K, rows, cols)).astype(np.float32)
    ct = torch.from_numpy(c).cuda()
    for got, w in ((bank.reconstruct(ct), True), (bank.adjoint(ct), False)):
        want = np.stack([T.reconstruct_natural(b.astype(np.float64), G, w) for b in c]).real
        assert np.abs(got.cpu().numpy() - want).max() <= 1e-5 * np.abs(want).max()
