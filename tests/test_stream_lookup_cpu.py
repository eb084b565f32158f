"""The stream of a call that names none: torch's current one if torch is in use,
the default one if torch is not there, or only just being imported.
"""

import sys
import types

import paper_1802_03084_gb300 as rf


def test_torch_absent_or_half_imported(monkeypatch):
    torch = types.ModuleType("torch")
    monkeypatch.setitem(sys.modules, "torch", torch)
    assert rf._stream(None) is None
    torch.cuda = types.ModuleType("torch.cuda")
    assert rf._stream(None) is None
    torch.cuda.is_initialized = lambda: False
    assert rf._stream(None) is None
    torch.cuda.is_initialized = lambda: True
    torch.cuda.current_stream = lambda: types.SimpleNamespace(cuda_stream=7)
    assert rf._stream(None) == 7
    monkeypatch.delitem(sys.modules, "torch")
    assert rf._stream(None) is None
