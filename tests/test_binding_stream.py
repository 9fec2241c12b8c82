"""The stream that the binding passes when none is given (no GPU: torch's CUDA state is stood in for)."""
import types

import pytest

torch = pytest.importorskip("torch")


@pytest.fixture()
def pm(monkeypatch):
    from paper_1610_10061_gb300 import build
    build.build()
    from paper_1610_10061_gb300 import pm as _pm
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=4321))
    return _pm


def test_the_raw_handle_of_the_current_device(pm, monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 100 + device, raising=False)
    assert pm._stream(None) == 103
    assert pm._stream(77) == 77


@pytest.mark.parametrize("how", ["gone", "raises"])
def test_without_the_private_names_the_public_call(pm, monkeypatch, how):
    def fail(*args):
        raise TypeError("another signature")

    if how == "gone":
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    else:
        monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 0, raising=False)
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", fail, raising=False)
    assert pm._stream(None) == 4321


def test_no_cuda_no_stream(pm, monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: False)
    assert pm._stream(None) == 0
