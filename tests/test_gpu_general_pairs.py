"""Parity of the two-stage register kernels (csrc/general_pairs.cuh) with the FP64
oracle at every length they are compiled for: all products of two radices, and
Bluestein lengths at both ends of each convolution length's range.  Each length
is tried as the rows of a plane with an odd number of rows and as its columns (a
ragged last column block), through real and complex banks, batches that end
inside a CTA, thresholds, masks and bfloat16.  Error measure and tolerances as in
test_gpu_general.py: max |gpu - oracle| / max |oracle| <= 1e-5 (bfloat16 1e-2)."""

import numpy as np
import pytest

from oracle import transform as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RADICES = (8, 10, 12, 15, 16, 20, 24, 25, 30, 32)
DIRECT = sorted({a * b for a in RADICES for b in RADICES})
# ends of the ranges of P = 128, 192, 256, 320, 400, 512, 640, 800, 1024 among the
# lengths with a prime factor above 7; 517 and 521 lie beyond (general.cu)
CHIRP = (11, 13, 61, 66, 95, 99, 127, 131, 159, 163, 199, 202, 253, 258, 319, 323, 397, 403, 511,
         517, 521)
TOL32, TOL16 = 1e-5, 1e-2


def _rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def _bank(rows, cols, cplx, rng):
    from paper_2006_04591_gb300.shearlet import Bank
    g = rng.standard_normal((2, rows, cols))
    if not cplx:
        g = 0.5 * (g + np.roll(g[:, ::-1, ::-1], (1, 1), (1, 2)))
    G = np.fft.fft2(g, axes=(-2, -1)) / np.sqrt(rows * cols)
    Wp = np.sum(np.abs(G) ** 2, axis=0)
    fill = np.sqrt(1.1 * Wp.max() - Wp)[None].astype(G.dtype)   # makes W constant
    G = np.concatenate([G, fill]) if cplx else np.concatenate([G, fill]).real
    make = Bank.from_complex_spectra if cplx else Bank.from_spectra
    return G, make(G, device=0)


@pytest.mark.parametrize("L", DIRECT + list(CHIRP))
@pytest.mark.parametrize("axis", ["rows", "cols"])
def test_lengths(L, axis):
    rng = np.random.default_rng(L)
    rows, cols = (L, 9) if axis == "cols" else (7, L)
    cplx = bool((L // 2 + (axis == "cols")) % 2)
    G, bank = _bank(rows, cols, cplx, rng)
    assert bank.general
    B = 3
    x = rng.standard_normal((B, rows, cols)).astype(np.float32)
    xt = torch.from_numpy(x).cuda()
    W = np.sum(np.abs(G) ** 2, axis=0)
    dec = lambda v, H: np.stack([T.decompose_natural(b.astype(np.float64), H) for b in v]).real
    rec = lambda v, w: np.stack([T.reconstruct_natural(b.astype(np.float64), G, w) for b in v]).real
    c = bank.decompose(xt)
    assert _rel(c.cpu().numpy(), dec(x, G)) <= TOL32
    assert _rel(bank.decompose(xt, dual=True).cpu().numpy(), dec(x, G / W)) <= TOL32
    cc = rng.standard_normal(c.shape).astype(np.float32)
    ct = torch.from_numpy(cc).cuda()
    assert _rel(bank.reconstruct(ct).cpu().numpy(), rec(cc, True)) <= TOL32
    th = np.full((B, bank.K), 0.7, np.float32)
    tht = torch.from_numpy(th).cuda()
    kept = np.where(np.abs(cc) >= 0.7, cc, 0.0)
    assert _rel(bank.adjoint(ct, thresh=tht).cpu().numpy(), rec(kept, False)) <= TOL32
    cb = bank.decompose(xt, dtype=torch.bfloat16)
    assert _rel(cb.float().cpu().numpy(), dec(x, G)) <= TOL16
    assert _rel(bank.reconstruct(cb).cpu().numpy(), rec(cb.float().cpu().numpy(), True)) <= TOL32
    mask = (rng.random(x.shape) < 0.5).astype(np.uint8)
    fe = rng.standard_normal(x.shape).astype(np.float32)
    u = torch.from_numpy(np.where(mask, x, fe)).cuda()
    got = bank.shrink(xt, tht, mask_u8=torch.from_numpy(mask).cuda(), f_est=torch.from_numpy(fe).cuda())
    # the fused pass and the separate ones run the same operations: equal bits
    assert torch.equal(got, bank.reconstruct(bank.decompose(u), thresh=tht))
    # one image alone and in the batch: the pairing of rows is per plane
    assert torch.equal(bank.decompose(xt[1:2].clone())[0], c[1])
