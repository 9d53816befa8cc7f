"""The Python binding's own decisions: the current stream's handle with and without torch's
raw-handle getters, and the type of the tensors a Synthesizer returns."""
import types

import pytest
import torch

import paper_2506_15183_gb300 as yoro


@pytest.mark.parametrize("missing", [(), ("_cuda_getCurrentRawStream",), ("_cuda_getDevice",)])
def test_current_stream_needs_no_private_getter(monkeypatch, missing):
    """A torch without the raw getters (private names) takes the public way to the same handle."""
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: types.SimpleNamespace(cuda_stream=77))
    for name, value in (("_cuda_getCurrentRawStream", lambda d: 70 + d), ("_cuda_getDevice", lambda: 7)):
        if name in missing:
            monkeypatch.delattr(torch._C, name, raising=False)
        else:
            monkeypatch.setattr(torch._C, name, value, raising=False)
    assert yoro._stream(None) == 77
    assert yoro._stream(5) == 5


class Frame(torch.Tensor):
    """A tensor subclass, as image libraries make them."""


@pytest.mark.gpu
def test_synthesizer_returns_plain_tensors_for_a_subclass():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_15183_gb300 import scene

    cfg = scene.small_config()
    c, d, _ = scene.render(cfg, 1)
    color, depth = torch.from_numpy(c).cuda(), torch.from_numpy(d).cuda()
    syn = yoro.Synthesizer(**cfg.camera())
    want = syn(color, depth)
    got = syn(color.as_subclass(Frame), depth)
    for a, b in zip(got, want):
        assert type(a) is torch.Tensor
        assert torch.equal(a, b)
    syn.close()
