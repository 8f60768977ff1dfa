"""Where the binding takes the current stream from: torch's raw lookups where it has them, its public interface otherwise."""
import torch

from paper_2604_16498_b200 import binding


class _Stream:
    cuda_stream = 77


def test_a_torch_without_the_raw_lookups_gets_the_public_one(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: _Stream)
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        with monkeypatch.context() as m:
            m.delattr(torch._C, name, raising=False)
            assert binding._find_raw_stream()() == 77


def test_the_raw_lookups_are_asked_for_the_current_device(monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 3, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda dev: 100 + dev, raising=False)
    assert binding._find_raw_stream()() == 103
