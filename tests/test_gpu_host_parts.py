"""Host-buffer frames that are copied and synthesized in parts (page-locked memory, two or
more parts): the bytes of the same frame synthesized on the device, for several part counts,
kernel heights, streams, pageable buffers, and a captured call that is replayed (needs a GPU)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def yoro():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_15183_gb300 as y
    from paper_2506_15183_gb300 import _build, scene

    _build.build_cuda()
    scene.build()
    y.load_library()
    return y


def _case(w, h, seed):
    from paper_2506_15183_gb300 import scene

    cfg = scene.quest_config().replace(w=w, h=h, n_prims=60)
    c, d, _ = scene.render(cfg, seed)
    return cfg, torch.from_numpy(c), torch.from_numpy(d)


@pytest.mark.parametrize("w,h,rows,pin", [(1501, 1499, 3, True), (1832, 1920, 3, True), (2064, 2208, 7, True),
                                           (9000, 300, 3, True), (300, 9001, 5, True), (1832, 1920, 3, False)])
def test_host_parts(yoro, w, h, rows, pin):
    cfg, c, d = _case(w, h, w + h)
    syn = yoro.Synthesizer(**cfg.camera(), kernel_rows=rows)
    ref, rmask = syn(c.cuda(), d.cuda())
    if pin:
        c, d = c.pin_memory(), d.pin_memory()
    out = torch.zeros((h, w, 4), dtype=torch.uint8, pin_memory=pin)
    mask = torch.zeros((h, w), dtype=torch.uint8, pin_memory=pin)
    side = torch.cuda.Stream()
    for stream in (None, side):
        out.zero_()
        mask.zero_()
        yoro.yoro_synthesize_host(syn.handle, c, d, out, mask, stream)
        (stream or torch.cuda.current_stream()).synchronize()
        assert torch.equal(out, ref.cpu()) and torch.equal(mask, rmask.cpu())
    if pin:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            yoro.yoro_synthesize_host(syn.handle, c, d, out, mask)
        out.zero_()
        mask.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref.cpu()) and torch.equal(mask, rmask.cpu())
    syn.close()
