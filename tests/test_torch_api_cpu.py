"""Simulator's use of PyTorch, without a GPU."""
import torch

from paper_2603_02804_gb300.torch_api import Simulator


def test_stream_without_the_raw_handle_call(monkeypatch):
    """A PyTorch without the private raw-stream call: the public stream object
    of the simulator's device."""
    asked = []
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device: asked.append(device) or "stream")
    sim = object.__new__(Simulator)
    sim.device, sim.handle = torch.device("cuda:1"), None
    assert sim._stream() == "stream" and asked == [torch.device("cuda:1")]


def test_stream_of_the_device(monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda i: 100 + i, raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    sim = object.__new__(Simulator)
    sim.handle = None
    for device, handle in (("cuda:1", 101), ("cuda", 103)):
        sim.device = torch.device(device)
        assert sim._stream() == handle
