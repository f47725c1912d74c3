"""The binding's current-stream handle (CPU, with stand-ins for PyTorch): a
stream that is given, the private raw-handle call, and a PyTorch without it."""
import types

from paper_2101_05617_gb300 import swepi


def _fake(with_raw):
    cuda = types.SimpleNamespace(current_device=lambda: 1,
                                 current_stream=lambda: types.SimpleNamespace(cuda_stream=0x77))
    c = types.SimpleNamespace(_cuda_getCurrentRawStream=lambda d: 0x50 + d) if with_raw else types.SimpleNamespace()
    return types.SimpleNamespace(cuda=cuda, _C=c)


def test_stream_handles(monkeypatch):
    assert swepi._stream(types.SimpleNamespace(cuda_stream=0x33)).value == 0x33
    for with_raw, want in ((True, 0x51), (False, 0x77)):
        monkeypatch.setattr(swepi, "_torch_module", _fake(with_raw))
        assert swepi._stream(None).value == want
