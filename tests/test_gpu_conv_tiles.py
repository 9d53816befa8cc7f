"""The one-tile convolution form where a CTA takes two 128-pixel tiles, the halo form where a CTA
walks several bands, and the network's half-resolution inputs (needs a GPU).

Layers against 64-bit sums: before rounding, the tensor core's FP32 accumulation of K exact
products in steps of 16 is within 2^-23 (K / 16 + 16) sum|p_i| (each addition within one unit
in the last place of a partial sum; a step's own sum within 16 of them), then the bias is
added and the result rounded to bfloat16."""
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


def _conv64(x, w):
    T, H, W, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    return sum(xp[:, dy:dy + H, dx:dx + W] @ w[:, dy, dx].t() for dy in range(3) for dx in range(3))


# A CTA takes two tiles from 2 SMs' worth of 128-pixel tiles on: 8x8 images pair up in a tile, so
# 4 SMs + 2 of them are an odd number of tiles, the last CTA half empty
@pytest.mark.parametrize("T,side,cin,cout,up", [
    ((4, 0), 8, 64, 256, False),
    ((4, 2), 8, 128, 256, False),
    ((4, 2), 8, 256, 256, True),
    ((4, 2), 8, 32, 64, False),     # 32 channels per step
    ((4, -2), 8, 64, 128, True),    # one tile per CTA, more CTAs than SMs
    ((2, 16), 16, 384, 128, False),  # halo form, several bands per CTA
    ((2, 15), 16, 128, 128, True),
])
def test_large_grids_match_64_bit_sums(un, T, side, cin, cout, up):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    T = T[0] * sms + T[1]
    g = torch.Generator(device="cuda").manual_seed(side + cin + cout)
    x = torch.rand((T, side, side, cin), generator=g, device="cuda").to(torch.bfloat16)
    wk = (torch.randn((cout, 9 * cin), generator=g, device="cuda") * (2.0 / (9 * cin)) ** 0.5).to(torch.bfloat16)
    b = torch.randn((cout,), generator=g, device="cuda") * 0.05
    f, cy, coff = 2 if up else 1, cout + 32, 32
    y = torch.full((T, f * side, f * side, cy), 7.0, dtype=torch.bfloat16, device="cuda")
    un.conv3x3(x, wk, b, y, y_coff=coff, upsample=up)
    assert un.status() == 0
    assert torch.all(y[..., :coff] == 7.0)
    w = wk.double().view(cout, 3, 3, cin)
    z = torch.relu(_conv64(x.double(), w) + b.double())
    absum = _conv64(x.double().abs(), w.abs())
    if up:
        z, absum = (a.repeat_interleave(2, 1).repeat_interleave(2, 2) for a in (z, absum))
    got = y[..., coff:].double()
    big = torch.maximum(z.abs(), got.abs()).clamp(min=2.0 ** -126)
    half_step = torch.exp2(torch.floor(torch.log2(big)) - 8)
    tol = 2.0 ** -23 * (9 * cin / 16 + 16) * absum * (1 + 2.0 ** -7) + 2.0 ** -23 * big + half_step
    bad = (got - z).abs() > tol
    assert not bad.any(), f"{int(bad.sum())} of {bad.numel()} outside the bound"


@pytest.mark.parametrize("T", [1, 3, 39, 610])
def test_network_equals_its_layers_on_concatenated_inputs(un, T):
    """The network reads the lower decoder levels at their own resolution and pools and colors in
    the convolutions' epilogues; the same layers one by one, on concatenated and upsampled
    tensors, give the same activations, so the colors differ by the exponential's and the
    division's roundings alone (8 units in the last place of 1)."""
    from paper_2506_15183_gb300 import weights as W

    flat = W.load_flat()
    p = W.split(flat)
    g = torch.Generator(device="cuda").manual_seed(T)
    x = torch.zeros((T, 64, 64, 32), dtype=torch.bfloat16, device="cuda")
    x[..., :6] = torch.rand((T, 64, 64, 6), generator=g, device="cuda")
    net = un.Inpainter(flat, max_tiles=T)
    rgb = torch.empty((T, 64, 64, 3), device="cuda")
    net.forward(x, rgb)
    assert un.status() == 0
    net.close()

    even = T + T % 2  # the 8x8 level pairs its images

    def conv(name, a):
        w = p[name + ".w"]
        cout = w.shape[0]
        wk = torch.from_numpy(un.kmajor(np.asarray(w, np.float32))).cuda().to(torch.bfloat16)
        y = torch.empty((even, a.shape[1], a.shape[2], cout), dtype=torch.bfloat16, device="cuda")
        un.conv3x3(a.contiguous(), wk, torch.from_numpy(np.asarray(p[name + ".b"], np.float32)).cuda(), y)
        return y

    def pool(a):
        return a.view(even, a.shape[1] // 2, 2, a.shape[2] // 2, 2, -1).amax((2, 4))

    def up(a):
        return a.repeat_interleave(2, 1).repeat_interleave(2, 2)

    a = torch.cat([x, x[:even - T]]) if even > T else x
    skips = []
    for lvl in range(4):
        a = conv(f"enc{lvl}b", conv(f"enc{lvl}a", pool(a) if lvl else a))
        skips.append(a)
    for lvl in (2, 1, 0):
        a = conv(f"dec{lvl}b", conv(f"dec{lvl}a", torch.cat([skips[lvl], up(a)], -1)))
    wo = torch.from_numpy(np.asarray(p["out.w"], np.float32).reshape(3, 32)).cuda().to(torch.bfloat16).float()
    bo = torch.from_numpy(np.asarray(p["out.b"], np.float32)).cuda()
    v = a[:T].float()
    acc = torch.zeros((T, 64, 64, 3), device="cuda")
    for c in range(32):
        acc = acc + v[..., c:c + 1] * wo[:, c]
    want = 1.0 / (1.0 + torch.exp(-(acc + bo)))
    assert un.status() == 0
    assert (rgb - want).abs().max() <= 2.0 ** -21
