"""The stream of a call (api._stream_handle) against a stand-in for torch: no GPU needed."""
import types

import pytest

from paper_1612_01799_gb300 import api


def fake(initialized, raw):
    cuda = types.SimpleNamespace(is_initialized=lambda: initialized, current_device=lambda: 3,
                                 current_stream=lambda: types.SimpleNamespace(cuda_stream=77))
    return types.SimpleNamespace(cuda=cuda, _C=types.SimpleNamespace(**raw))


@pytest.mark.parametrize("initialized,raw,want", [
    (True, {"_cuda_getCurrentRawStream": lambda dev: 100 + dev}, 103),
    (False, {"_cuda_getCurrentRawStream": lambda dev: 100 + dev}, 77),
    (True, {}, 77),                       # a torch build without the private function
])
def test_current_stream(monkeypatch, initialized, raw, want):
    monkeypatch.setattr(api, "_torch_module", fake(initialized, raw))
    assert api._stream_handle(None) == want


def test_given_stream():
    assert api._stream_handle(types.SimpleNamespace(cuda_stream=5)) == 5
