"""The weight gradient of the inpainter's 3x3 layers (csrc/conv_dw.cu) against 64-bit sums
(needs a GPU), through the library's internal entry and through training steps.

Products of bfloat16 values are exact in FP32.  An element's sum runs through at most side / 2
tensor-core additions per box of 8 rows (16 pixels each) and one FP32 addition per box and
share, each within one unit in the last place (2^-23) of a partial sum, itself at most
sum|p|: |gpu - exact| <= 2^-23 (side / 2 + boxes) sum|p|."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# the levels' layers: side, input channels, their channel stride, output channels
LAYERS = [(64, 6, 32, 32), (64, 96, 96, 32), (32, 32, 32, 64), (32, 192, 192, 64), (16, 384, 384, 128),
          (8, 128, 128, 256), (8, 256, 256, 256)]


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


def _conv_dw(dz, x, cin):
    """yoro::conv_dw_launch (csrc/unet_internal.h) on torch tensors."""
    import paper_2506_15183_gb300 as yoro

    lib, P, I = yoro.load_library(), ctypes.c_void_p, ctypes.c_int
    launch = getattr(lib, "_ZN4yoro14conv_dw_launchEPKvS1_iiiiiiPfS2_P11CUstream_st")
    launch.argtypes, launch.restype = [P, P] + 6 * [I] + [P, P, P], I
    size = getattr(lib, "_ZN4yoro17conv_dw_workspaceEi")
    size.argtypes, size.restype = [I], ctypes.c_size_t
    sms = getattr(lib, "_ZN4yoro8sm_countEv")()
    T, side, _, cout = dz.shape
    ws = torch.empty(size(sms) // 4, device="cuda")
    dw = torch.full((cout, cin, 3, 3), float("nan"), device="cuda")
    rc = launch(dz.data_ptr(), x.data_ptr(), x.shape[3], T, side, cin, cout, sms, ws.data_ptr(), dw.data_ptr(),
                torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    return dw


def _exact(dz, x, cin):
    T, side, _, cout = dz.shape
    xp = torch.nn.functional.pad(x[..., :cin].double(), (0, 0, 1, 1, 1, 1))
    z = dz.double().reshape(-1, cout).t()
    w = torch.empty((cout, cin, 3, 3), dtype=torch.float64, device="cuda")
    for dy in range(3):
        for dx in range(3):
            w[:, :, dy, dx] = z @ xp[:, dy:dy + side, dx:dx + side].reshape(-1, cin)
    return w


def _layer(T, side, cin, xcs, cout, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((T, side, side, xcs), generator=g, device="cuda").clamp(min=0)
    x[..., cin:] = 0
    dz = torch.randn((T, side, side, cout), generator=g, device="cuda")
    return dz.to(torch.bfloat16), x.to(torch.bfloat16)


# 2 tiles: one box per CTA or fewer boxes than CTAs; 6: uneven shares; 38 and 64: rings refilled
@pytest.mark.parametrize("T", [2, 6, 38, 64])
@pytest.mark.parametrize("side,cin,xcs,cout", LAYERS)
def test_weight_gradient_matches_64_bit_sums(un, T, side, cin, xcs, cout):
    dz, x = _layer(T, side, cin, xcs, cout, T + side + cin)
    got = _conv_dw(dz, x, cin)
    want, absum = _exact(dz, x, cin), _exact(dz.abs(), x.abs(), cin)
    bound = 2.0 ** -23 * (side / 2 + T * side / 8) * absum
    bad = (got.double() - want).abs() > bound
    assert not bad.any(), f"{int(bad.sum())} of {bad.numel()} outside the bound"
    assert torch.equal(got, _conv_dw(dz, x, cin))  # the same bits on every run
    assert un.status() == 0


# relative L2 error against 64 bits of FP32 fused multiply-adds in chains of at most 4096
# pixels, measured on these inputs: dense ones, and sparse gradients on non-negative inputs
@pytest.mark.parametrize("T,side,cin,xcs,cout,dense,sparse", [
    (4, 64, 6, 32, 32, 2.9e-7, 2.7e-7), (4, 64, 96, 96, 32, 2.9e-7, 2.6e-7), (4, 32, 192, 192, 64, 1.3e-7, 8.9e-8),
    (4, 16, 384, 384, 128, 1.1e-7, 5.5e-8), (4, 8, 128, 128, 256, 9.7e-8, 3.8e-8), (4, 8, 256, 256, 256, 9.7e-8, 4.1e-8),
    (64, 64, 6, 32, 32, 4.5e-7, 4.2e-7), (64, 64, 96, 96, 32, 3.8e-7, 3.1e-7), (64, 32, 32, 32, 64, 3.1e-7, 2.8e-7),
    (64, 32, 192, 192, 64, 2.9e-7, 1.7e-7), (64, 16, 384, 384, 128, 2.5e-7, 1.1e-7),
    (64, 8, 128, 128, 256, 1.2e-7, 8.5e-8), (64, 8, 256, 256, 256, 1.6e-7, 7.8e-8)])
def test_weight_gradient_is_no_less_precise_than_fp32_multiply_adds(un, T, side, cin, xcs, cout, dense, sparse):
    for limit in (dense, sparse):
        g = torch.Generator(device="cuda").manual_seed(T + side + cin)
        x = torch.randn((T, side, side, xcs), generator=g, device="cuda")
        if limit == sparse:
            x = x.clamp(min=0)
        x[..., cin:] = 0
        dz = torch.randn((T, side, side, cout), generator=g, device="cuda")
        if limit == sparse:
            dz = dz * (torch.rand((T, side, side, cout), generator=g, device="cuda") < 0.15)
            dz = dz * torch.exp(torch.randn((T, side, side, 1), generator=g, device="cuda"))
        dz, x = dz.to(torch.bfloat16), x.to(torch.bfloat16)
        want = _exact(dz, x, cin)
        err = float((_conv_dw(dz, x, cin).double() - want).norm() / want.norm())
        assert err <= limit, (err, limit)


@pytest.mark.parametrize("side,cin,xcs,cout", [(64, 32, 32, 32), (32, 64, 64, 64), (16, 64, 64, 128), (8, 128, 128, 256)])
def test_infinite_activations_reach_the_taps_they_meet_and_no_others(un, side, cin, xcs, cout):
    """An infinite input in the first column is never under a tap to its right (no gradient pixel
    lies left of the image), nor one in the last column under a tap to its left."""
    dz, x = _layer(3, side, cin, xcs, cout, side)
    want = _conv_dw(dz, x.clone().index_fill_(3, torch.tensor([0, 33 % cin], device="cuda"), 0.0), cin)
    y = x.clone()
    y[..., 0] = 0
    y[..., 33 % cin] = 0
    y[1, 5, 0, 0] = float("inf")
    y[1, 5, side - 1, 33 % cin] = float("inf")
    got = _conv_dw(dz, y, cin)
    w64 = _exact(dz, y, cin)
    assert torch.equal(torch.isfinite(got), torch.isfinite(w64))
    fine = torch.isfinite(w64)
    assert torch.equal(got[fine], want[fine])
    assert not fine[:, 0, :, :2].any() and fine[:, 0, :, 2].all()


def test_training_step_with_infinite_inputs(un):
    """The same through a training step: a tile whose first column holds an infinity and which has
    no hole leaves the gradient of the taps that never meet it as they are without the tile's
    infinity."""
    from paper_2506_15183_gb300 import weights as W

    g = torch.Generator(device="cuda").manual_seed(2)
    x = torch.zeros((2, 64, 64, 32), device="cuda")
    x[..., :6] = torch.rand((2, 64, 64, 6), generator=g, device="cuda")
    hole = torch.zeros((2, 64, 64), dtype=torch.uint8, device="cuda")
    hole[1, 20:40, 20:40] = 1
    gt = torch.randint(0, 256, (2, 64, 64, 3), generator=g, device="cuda", dtype=torch.uint8)
    flat = W.init_params(5)
    grads = []
    for v in (0.25, float("inf")):
        x[0, 31, 0, 0] = v
        tr = un.Trainer(flat, batch_tiles=2, lr=0.0)
        tr.step(x.to(torch.bfloat16), gt, hole)
        grads.append(W.split(tr.read("grads"))["enc0a.w"].reshape(32, 6, 3, 3))
        tr.close()
    assert un.status() == 0
    finite, inf = grads
    assert np.isfinite(finite).all()
    assert np.array_equal(inf[:, 1:], finite[:, 1:])
    assert np.array_equal(inf[:, 0, :, 2], finite[:, 0, :, 2])
