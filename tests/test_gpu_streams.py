"""The binding launches on torch's current stream of the tensors' device, and
refuses tensors that are not on one."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_current_stream_follows_the_context():
    from paper_2006_04591_gb300.shearlet import current_stream_ptr
    dev = torch.device("cuda", 0)
    side = torch.cuda.Stream()
    for d in (0, dev, torch.device("cuda")):
        assert current_stream_ptr(d) == torch.cuda.current_stream(0).cuda_stream
        with torch.cuda.stream(side):
            assert current_stream_ptr(d) == side.cuda_stream
    with pytest.raises(ValueError):
        current_stream_ptr(torch.device("cpu"))


def test_host_tensors_are_refused():
    from paper_2006_04591_gb300 import nn
    from paper_2006_04591_gb300.shearlet import Bank
    bank = Bank.create(32, 32, 1, device=0)
    c = torch.zeros((1, bank.K, 32, 32))
    with pytest.raises(ValueError):
        bank.reconstruct(c)
    with pytest.raises(ValueError):
        nn.prelu(torch.zeros(8), torch.zeros(1))


def test_repeated_calls_with_other_batches_and_streams():
    """Workspace sizes are kept per batch; work on two streams does not mix."""
    from paper_2006_04591_gb300.shearlet import Bank
    bank = Bank.create(64, 64, 2, device=0)
    g = torch.Generator(device="cuda").manual_seed(0)
    x = torch.randn((5, 64, 64), device="cuda", generator=g)
    want = bank.reconstruct(bank.decompose(x))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = []
    for k in range(6):
        with torch.cuda.stream(streams[k % 2]):
            n = 1 + k % 5
            outs.append((n, bank.reconstruct(bank.decompose(x[:n].contiguous()))))
    torch.cuda.synchronize()
    for n, y in outs:
        assert torch.equal(y, want[:n])
