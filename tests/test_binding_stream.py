"""The binding's device and stream with a torch that lacks the private calls it
prefers: the public ones serve."""
import importlib.util
import os
import types

import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_public_calls_serve(monkeypatch):
    for name in ("_cuda_getDevice", "_cuda_getCurrentRawStream"):
        monkeypatch.delattr(torch._C, name, raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda device=None: types.SimpleNamespace(cuda_stream=1000 + device))
    path = os.path.join(ROOT, "paper_2009_10917_gb300", "bs.py")
    spec = importlib.util.spec_from_file_location("paper_2009_10917_gb300.bs_again", path)
    bs = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bs)
    assert bs._stream() == 1003
