"""Argument marshalling across PyTorch builds: the current stream by the fast calls where this torch has them and by
the public one where not, and the errors of a Python without torch."""
import sys
import types

import numpy as np
import pytest

import paper_2302_14812_gb300 as rd


def _fake_torch(**fast):
    """A torch with CUDA whose current stream is 7 (0x77 by the fast calls)."""
    calls = []
    cuda = types.SimpleNamespace(is_available=lambda: True, is_initialized=lambda: bool(calls),
                                 init=lambda: calls.append("init"),
                                 current_stream=lambda: types.SimpleNamespace(cuda_stream=7))
    return types.SimpleNamespace(cuda=cuda, _C=types.SimpleNamespace(**fast)), calls


FAST = {"_cuda_getCurrentRawStream": lambda dev: 0x70 + dev, "_cuda_getDevice": lambda: 7}


@pytest.mark.parametrize("have,handle", [(tuple(FAST), 0x77), ((), 7), (("_cuda_getDevice",), 7),
                                         (("_cuda_getCurrentRawStream",), 7)])
def test_current_stream(monkeypatch, have, handle):
    t, calls = _fake_torch(**{k: FAST[k] for k in have})
    monkeypatch.setattr(rd, "_torch_mod", t)
    monkeypatch.setattr(rd, "_raw_stream", None, raising=False)
    assert rd._stream_ptr(None) == handle and rd._stream_ptr(None) == handle
    assert calls == ["init"]


def test_without_torch(monkeypatch):
    monkeypatch.setattr(rd, "_torch_mod", None)
    monkeypatch.setattr(rd, "_raw_stream", None, raising=False)
    monkeypatch.setitem(sys.modules, "torch", None)             # an import of torch raises ImportError
    assert rd._stream_ptr(None) is None
    keep = []
    assert rd._as_f64(np.zeros((2, 3)), keep)[1:] == (rd.RD_MEM_HOST, 6)
    d = object.__new__(rd.RadiationDetector)
    d.n_pix, d.n_bins = 2, 4
    with pytest.raises(ImportError):
        d.read("float32", "cuda")
