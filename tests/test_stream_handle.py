"""The current stream's handle comes from torch's raw entry where there is one, else from
the public call."""
import importlib
import sys

import torch

from paper_1703_04446_gb300 import lgnk


class _Stream:
    cuda_stream = 4711


def _fresh(monkeypatch):
    """lgnk imported anew, without touching the module the other tests hold."""
    import paper_1703_04446_gb300.lgnk as held
    import paper_1703_04446_gb300 as pkg
    monkeypatch.setattr(pkg, "lgnk", held)                       # both put back at the test's end
    monkeypatch.setitem(sys.modules, "paper_1703_04446_gb300.lgnk", held)
    del sys.modules["paper_1703_04446_gb300.lgnk"]
    return importlib.import_module("paper_1703_04446_gb300.lgnk")


def test_public_call_where_torch_has_no_raw_entry(monkeypatch):
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda index: _Stream())
    assert _fresh(monkeypatch)._raw_stream(0) == 4711


def test_raw_entry_where_there_is_one(monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: 42 + index, raising=False)
    assert _fresh(monkeypatch)._raw_stream(1) == 43


def test_the_held_module_is_back():
    import paper_1703_04446_gb300 as pkg
    assert sys.modules["paper_1703_04446_gb300.lgnk"] is pkg.lgnk is lgnk
