"""The Python binding's own decisions: the type of the tensors a Synthesizer returns."""
import pytest
import torch

import paper_2506_15183_gb300 as yoro


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
