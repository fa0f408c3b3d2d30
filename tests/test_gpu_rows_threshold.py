"""launch_rows_r2c_t (csrc/fast.cu), the library's forward row pass, applies the
thresholds it is given whether or not it is told that the rows are coefficients, and
refuses thresholds on masked input, which has none.  Called by its C++ symbol; against the
float64 row DFT of the thresholded rows (1e-5 of the largest)."""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SYMBOL = "_ZN3shl17launch_rows_r2c_tEiNS_6InModeEbPKvPKhPKfS6_P6float2iiPKS7_P11CUstream_stb"
IN_F32, IN_MASKED = 0, 2
TW_P = 4096


def _call(M, mode, x, mask, fest, th, out, coeffs):
    from paper_2006_04591_gb300 import shearlet as S
    f = getattr(S.lib(), SYMBOL)
    vp, i = ctypes.c_void_p, ctypes.c_int
    f.restype, f.argtypes = i, [i, i, ctypes.c_bool, vp, vp, vp, vp, vp, i, i, vp, vp, ctypes.c_bool]
    w = np.exp(-2j * np.pi * np.arange(TW_P) / TW_P).astype(np.complex64)
    tw = torch.from_numpy(w).cuda()
    p = lambda t: None if t is None else t.data_ptr()  # noqa: E731
    e = f(M, mode, th is not None, p(x), p(mask), p(fest), p(th), p(out), out.shape[2], out.shape[0],
          p(tw), S.current_stream_ptr(0), coeffs)
    torch.cuda.synchronize()
    return e


@pytest.mark.parametrize("M", [16, 64, 512, 1024])
@pytest.mark.parametrize("coeffs", [False, True])
@pytest.mark.parametrize("thresholds", [False, True])
def test_thresholds_are_applied(M, coeffs, thresholds):
    nsub, N = 3, 32
    g = torch.Generator(device="cuda").manual_seed(M)
    x = torch.randn((nsub, N, M), device="cuda", generator=g)
    th = torch.tensor([0.5, 0.0, 1.5], device="cuda") if thresholds else None
    out = torch.empty((nsub, M // 2 + 1, N), dtype=torch.complex64, device="cuda")
    assert _call(M, IN_F32, x, None, None, th, out, coeffs) == 0
    v = x.double()
    if thresholds:
        v = torch.where(v.abs() >= th.double()[:, None, None], v, 0.0)
    want = torch.fft.rfft(v).transpose(1, 2)
    assert (out - want).abs().max().item() <= 1e-5 * want.abs().max().item()


def test_masked_input_takes_no_thresholds():
    x, f = (torch.zeros((1, 32, 64), device="cuda") for _ in range(2))
    mask = torch.ones((1, 32, 64), dtype=torch.uint8, device="cuda")
    out = torch.empty((1, 33, 32), dtype=torch.complex64, device="cuda")
    assert _call(64, IN_MASKED, x, mask, f, None, out, False) == 0
    assert _call(64, IN_MASKED, x, mask, f, torch.ones(1, device="cuda"), out, False) != 0
