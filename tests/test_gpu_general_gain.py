"""The general path's rounding must not lean one way.  There and back, an image comes out
as (1 + g) x plus noise; g adds up the mean gain of eight line transforms whose roots are
rounded to float32.  Of a pair of Bluestein's transforms less than 2e-8 may be left per
line, 1.6e-7 in all, and 3e-8 is allowed for the rest.  Lengths: Bluestein's at both ends of each
convolution length (23 .. 61, 67 .. 127, 134 .. 254, 262 .. 509), among them primes and
multiples of 23 and 47, and lengths with factors of 11 to 19, which run direct stages."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [23, 29, 46, 61, 67, 94, 127, 134, 188, 254, 262, 307, 437, 502, 509,
                               55, 88, 220, 416, 440, 475])
def test_mean_gain(L):
    from paper_2006_04591_gb300 import synth
    from paper_2006_04591_gb300.shearlet import Bank
    ky, kx = np.fft.fftfreq(L)[:, None], np.fft.fftfreq(L)[None]
    low = np.exp(-(ky ** 2 + kx ** 2) / 0.02)
    bank = Bank.from_spectra(np.stack([low, np.sqrt(1.0 - low ** 2)]), device=0)
    x = np.stack([synth.cartoon(L, L, s) for s in range(8)]).astype(np.float32)
    xt = torch.from_numpy(x).cuda()
    y = bank.reconstruct(bank.decompose(xt)).double()
    xd = xt.double()
    gain = float(((y - xd) * xd).sum() / (xd * xd).sum())
    assert abs(gain) <= 1.9e-7
