"""General poses at widths whose band window fits shared memory without its words' largest
depths but not with them (needs a GPU): with up to 7 kernel rows the frame keeps the band fill,
two kernels after the clear, and its bytes are the oracle's."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def yoro():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_15183_gb300 as y
    from paper_2506_15183_gb300 import _build

    _build.build_cuda()
    y.load_library()
    return y


def _nodes(call):
    """Number of nodes (kernels and clears) that `call(stream)` enqueues, by capturing it."""
    rt = ctypes.CDLL("libcudart.so.13")
    P = ctypes.c_void_p
    rt.cudaStreamBeginCapture.argtypes = [P, ctypes.c_int]
    rt.cudaStreamEndCapture.argtypes = [P, ctypes.POINTER(P)]
    rt.cudaGraphGetNodes.argtypes = [P, P, ctypes.POINTER(ctypes.c_size_t)]
    rt.cudaGraphDestroy.argtypes = [P]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(s.cuda_stream, 2) == 0  # relaxed
    call(s)
    graph, n = P(), ctypes.c_size_t(0)
    assert rt.cudaStreamEndCapture(s.cuda_stream, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    rt.cudaGraphDestroy(graph)
    return n.value


# widest windows, with and without the maxima: 9248 / 9384 columns with 3 rows, 5544 / 5632 with
# 5, 3960 / 4016 with 7, 1848 / 1872 with 15 (whose frames between them take a gather pass)
@pytest.mark.parametrize("w,rows,nearest,nodes", [
    (9240, 3, False, 3), (9300, 3, False, 3), (9376, 3, False, 3), (9300, 3, True, 3), (5589, 5, False, 3),
    (3989, 7, True, 3), (1840, 15, False, 3), (1860, 15, False, 4), (1860, 15, True, 4)])
def test_frames_near_the_widest_window(yoro, w, rows, nearest, nodes):
    import oracle

    h = 21
    rng = np.random.default_rng(w + rows)
    depth = np.full((h, w), 40.0, np.float32) + rng.uniform(0, 1, (h, w)).astype(np.float32)
    for _ in range(5):
        x0, y0 = int(rng.integers(0, w)), int(rng.integers(0, h))
        depth[y0:y0 + 9, x0:x0 + w // 5] = np.float32(rng.uniform(0.3, 3.0))
    color = rng.integers(0, 256, (h, w, 4), dtype=np.uint8)
    rot = np.array([[0.9998, 0.0, -0.02], [0.0, 1.0, 0.0], [0.02, 0.0, 0.9998]], np.float32)
    pos, one = [0.063, 0.002, 0.0], np.float32
    syn = yoro.Synthesizer(w, h, w / 2, w / 2, w / 2, h / 2, 0.0, kernel_rows=rows, nearest_first=nearest, pose=(rot, pos))
    c, d = torch.from_numpy(color).cuda(), torch.from_numpy(depth).cuda()
    out, mask = syn(c, d)
    ref, rmask = oracle.synthesize_pose(color, depth, one(w / 2), one(w / 2), one(w / 2), one(h / 2), rot, pos,
                                        one(0.05), one(1000.0), kernel_rows=rows, nearest_first=nearest)
    assert np.array_equal(mask.cpu().numpy(), rmask)
    assert np.array_equal(out.cpu().numpy(), ref)
    n = _nodes(lambda s: yoro.yoro_synthesize(syn.handle, c, d, out, mask, s))
    assert n == nodes, f"{n} nodes, {nodes} expected: clear, scatter, band fill or gather and fill"
    syn.close()
