"""The binding's stream argument: no torch for a caller with a handle of its own, and torch's public call where the private
one is missing."""
import os
import subprocess
import sys
import types

import torch

from paper_2203_05705_b200 import ard

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_handle_needs_no_torch():
    code = ("import sys; from paper_2203_05705_b200 import ard; "
            "assert ard._stream(7) == 7 and ard._stream(type('S', (), {'cuda_stream': 9})()) == 9; "
            "assert 'torch' not in sys.modules")
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True)


def test_the_current_stream_with_and_without_the_private_name(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 40 + device, raising=False)
    monkeypatch.setattr(ard, "_current_stream", None)
    assert ard._stream(None) == 43
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=5))
    monkeypatch.setattr(ard, "_current_stream", None)
    assert ard._stream(None) == 5
