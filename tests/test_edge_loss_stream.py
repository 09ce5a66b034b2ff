"""Which pass EdgeLoss takes (CPU, no library call): the gradient is kept only where the scene's stream is
torch's current one on the device of the input, whatever device is current."""
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

import paper_2607_00579_gb300 as epo  # noqa: E402


@pytest.mark.parametrize("current_device", [0, 1])
@pytest.mark.parametrize("device,scene_stream,fused", [(0, 0, True), (1, 0, False), (1, 77, True), (0, 77, False)])
def test_stream_of_the_inputs_device(monkeypatch, current_device, device, scene_stream, fused):
    streams = {0: 0, 1: 77}  # device 1's current stream is a side stream; 0 is the default stream's handle
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", streams.__getitem__, raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: current_device)
    took = []
    monkeypatch.setattr(epo.EdgeLoss, "_fn", SimpleNamespace(apply=lambda xi, scene, f: took.append(f)))
    xi = SimpleNamespace(requires_grad=True, device=torch.device("cuda", device))
    epo.EdgeLoss.apply(xi, SimpleNamespace(refine=False, _stream=scene_stream))
    assert took == [fused]
