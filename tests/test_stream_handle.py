"""The stream that the binding enqueues on: the given one, else torch's current
one, by the public call where torch has no raw handle to give."""
import types

import pytest

import paper_2605_17230_gb300 as mld

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_without_the_raw_handle(monkeypatch, missing):
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda dev: 11, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 0, raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    assert mld._stream(5) == 5
    assert mld._stream(None) == 11
    monkeypatch.delattr(torch._C, missing)
    assert mld._stream(None) == 77
