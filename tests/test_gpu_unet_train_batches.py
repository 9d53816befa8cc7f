"""Training steps on batches whose passes take several turns of their grids (needs a GPU): the
gradient against 64-bit sums, and the same weight-gradient bits on a repeat and in a trainer
made for more tiles.

The reference rounds activations and layer gradients to bfloat16 as the kernels do, with
64-bit sums between, so the two differ where a sum lies at a rounding boundary and the step
travels on: 1.5e-3 to 1.2e-2 of the gradient's norm by batch.  Bounds: 3e-2 of the whole
gradient's norm, 0.1 of each tensor's; a pass that left out part of a batch would miss whole
tiles."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def un():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2506_15183_gb300 as yoro
    from paper_2506_15183_gb300 import _build
    from paper_2506_15183_gb300 import unet

    _build.build_cuda()
    yoro.load_library()
    return unet


def _step(un, flat, batch, batch_tiles):
    tr = un.Trainer(flat, batch_tiles=batch_tiles, lr=0.0)
    tr.step(*batch)
    grads, loss = tr.read("grads"), float(tr.read("loss")[0])
    assert un.status() == 0
    tr.close()
    return grads, loss


@pytest.mark.parametrize("T", [34, 64])
def test_gradient_of_a_large_batch(un, T):
    from paper_2506_15183_gb300 import weights as W
    from perf import cases

    x, hole, gt = cases._tiles(T, 100 + T)
    flat = W.init_params(T)
    grads, loss = _step(un, flat, (x, gt, hole), T)
    loss64, grads64 = cases._grads64(x[..., :6].double(), hole, gt, cases._params64(flat))
    want = grads64.cpu().numpy()
    assert abs(loss - loss64) <= 1e-3 * loss64
    assert np.linalg.norm(grads - want) <= 3e-2 * np.linalg.norm(want)
    got, ref = W.split(grads), W.split(want)
    for key in ref:
        assert np.linalg.norm(got[key] - ref[key]) <= 0.1 * np.linalg.norm(ref[key]), key
    again, _ = _step(un, flat, (x, gt, hole), T + 30)
    more = W.split(again)
    for name, shape, _ in W.layers():
        if len(shape) == 4:
            assert np.array_equal(got[name + ".w"], more[name + ".w"]), name
