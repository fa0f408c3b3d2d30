"""The two-stage kernels carry an image's partial sums from one chunk of subbands to the
next when the staging area holds fewer than K: staging areas of two and of five planes,
odd and even numbers of subbands, direct lengths (80, 96) and Bluestein's (46, 253) as rows
and as columns, real and complex filters.  The area is read from the environment once per
process.  Error measure and tolerance as in test_gpu_general.py (1e-5 of the largest);
the fused shrink equals the separate passes bit by bit."""

import os
import subprocess
import sys
import textwrap

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = textwrap.dedent("""
    import sys
    rows, cols, K, cplx = (int(a) for a in sys.argv[1:5])
    sys.path.insert(0, %r)
    import numpy as np, torch
    from oracle import transform as T
    from paper_2006_04591_gb300.shearlet import Bank
    rng = np.random.default_rng(rows + K)
    g = rng.standard_normal((K - 1, rows, cols))
    if not cplx:
        g = 0.5 * (g + np.roll(g[:, ::-1, ::-1], (1, 1), (1, 2)))
    G = np.fft.fft2(g, axes=(-2, -1)) / np.sqrt(rows * cols)
    Wp = np.sum(np.abs(G) ** 2, axis=0)
    G = np.concatenate([G, np.sqrt(1.1 * Wp.max() - Wp)[None].astype(G.dtype)])   # W constant
    bank = Bank.from_complex_spectra(G) if cplx else Bank.from_spectra(G.real)
    assert bank.general
    G = G if cplx else G.real
    B = 3
    rel = lambda a, b: np.abs(a.cpu().numpy() - b).max() / np.abs(b).max()
    x = torch.from_numpy(rng.standard_normal((B, rows, cols)).astype(np.float32)).cuda()
    c = bank.decompose(x)
    want = np.stack([T.decompose_natural(v.astype(np.float64), G) for v in x.cpu().numpy()]).real
    e = [rel(c, want)]
    cc = torch.from_numpy(rng.standard_normal(tuple(c.shape)).astype(np.float32)).cuda()
    for f, w in ((bank.reconstruct, True), (bank.adjoint, False)):
        want = np.stack([T.reconstruct_natural(v.astype(np.float64), G, w) for v in cc.cpu().numpy()]).real
        e.append(rel(f(cc), want))
    th = torch.full((B, K), 0.3, device="cuda")
    same = torch.equal(bank.shrink(x, th), bank.reconstruct(c, thresh=th))
    print(e, same)
    assert max(e) <= 1e-5 and same
""" % ROOT)


@pytest.mark.parametrize("planes", [2, 5])
@pytest.mark.parametrize("rows,cols,K,cplx", [(80, 96, 17, 0), (96, 80, 6, 1), (253, 96, 7, 0),
                                              (80, 253, 4, 0), (46, 46, 9, 1)])
def test_partial_sums_between_chunks(rows, cols, K, cplx, planes):
    mb = (planes + 0.5) * rows * (cols // 2 + 1) * 8 / 2 ** 20
    r = subprocess.run([sys.executable, "-c", SCRIPT, str(rows), str(cols), str(K), str(cplx)],
                       env=dict(os.environ, SHL_STAGE_MB=repr(mb)), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
