"""shl_nn_gate_forward on bfloat16 coefficients, which the Python gate does not pass: four
values per load (plane sizes that are multiples of 4, 16-byte aligned) and one, against
float64 (2e-5 of the largest, as in test_gpu_elementwise.py) and against the same call on the
coefficients as float32, whose arithmetic is the same (2e-6)."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("HW", [1, 4, 7, 9, 64, 1020, 1021, 4096, 262144])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("scaled", [False, True])
def test_gate_forward_bf16(HW, shift, scaled):
    from paper_2006_04591_gb300 import nn
    g = torch.Generator(device="cuda").manual_seed(HW)
    B, K, tau = 2, 3, 0.1
    n = B * K * HW
    c = torch.randn(n + shift, device="cuda", generator=g).to(torch.bfloat16)[shift:]
    d = torch.rand(B * K, device="cuda", generator=g) + 0.3
    s = torch.rand(K, device="cuda", generator=g) + 0.5 if scaled else None

    def run(c, is_bf16):
        y = torch.full((n,), float("nan"), device="cuda")
        nn._chk("gate_forward", nn.lib().shl_nn_gate_forward(
            c.data_ptr(), is_bf16, d.data_ptr(), None if s is None else s.data_ptr(), K, tau,
            y.data_ptr(), B * K, HW, nn._st(y)))
        return y

    got, same = run(c, 1), run(c.float(), 0)
    assert (got - same).abs().max().item() <= 2e-6 * same.abs().max().item()
    lim = (d * s.repeat(B) if scaled else d).double()[:, None]
    v = c.double().reshape(B * K, HW)
    want = v * torch.sigmoid((v.abs() / lim - 1.0) / tau)
    err = (got.double().reshape(B * K, HW) - want).abs().max().item()
    assert err <= 2e-5 * want.abs().max().item()
