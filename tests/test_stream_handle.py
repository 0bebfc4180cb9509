"""The binding's stream argument: torch's current stream when none is given, with
torch's raw lookups and without them (they are not part of torch's public
interface)."""
import pytest

from paper_2311_01598_gb300 import ks


class _Stream:
    cuda_stream = 0x1230


@pytest.mark.parametrize("missing", [(), ("_cuda_getCurrentRawStream",), ("_cuda_getDevice",),
                                     ("_cuda_getCurrentRawStream", "_cuda_getDevice")])
def test_current_stream(monkeypatch, missing):
    torch = pytest.importorskip("torch")
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: _Stream())
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 0x1000 + 0x230 * (d == 3), raising=False)
    for name in missing:
        monkeypatch.delattr(torch._C, name)
    monkeypatch.setattr(ks, "_current_stream", None)
    assert ks._stream_handle(None).value == 0x1230
    assert ks._stream_handle(None).value == 0x1230


def test_given_stream():
    assert ks._stream_handle(_Stream()).value == 0x1230
    assert ks._stream_handle(0x40).value == 0x40
