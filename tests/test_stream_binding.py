"""The binding's current stream in a torch with and without the raw call (no GPU needed:
both are stand-ins)."""

import types

import pytest

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("raw", [True, False])
def test_current_stream_ptr(monkeypatch, raw):
    from paper_2006_04591_gb300.shearlet import current_stream_ptr
    asked = []
    if raw:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda i: asked.append(i) or 77, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
        monkeypatch.setattr(torch.cuda, "current_stream",
                            lambda i: asked.append(i) or types.SimpleNamespace(cuda_stream=77))
    assert current_stream_ptr(torch.device("cuda", 3)) == 77 and current_stream_ptr(1) == 77
    assert asked == [3, 1]
    with pytest.raises(ValueError):
        current_stream_ptr(torch.device("cpu"))
