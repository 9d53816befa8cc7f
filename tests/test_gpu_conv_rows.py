"""The row form of the inpainter's 3x3 convolution (csrc/conv_rows.cu) at the sizes where its
units, image groups and masks end, against 64-bit sums (needs a GPU).

Before rounding, the tensor core's FP32 accumulation is within 2 K u sum|p_i| of the exact
sum (u = 2^-24, K products; one unit in the last place per addition), then the bias is added
and the result rounded to bfloat16, so |gpu - exact| <= 2 K u sum|p| (1 + 2^-7) + ulp_f32 +
half a bfloat16 step of the larger of the two."""
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


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


# rows of a unit are 256 / Cout, fewer while that leaves SMs idle; a group is 128 / W images
@pytest.mark.parametrize("T,H,W,cin,cout,up,relu", [
    (1, 64, 64, 32, 32, False, True),     # one image of a group of two, two-row units
    (3, 64, 64, 96, 32, False, True),     # a half-empty last group, three channel blocks
    (39, 64, 64, 32, 32, False, True),    # eight-row units, odd image count
    (20, 64, 64, 32, 32, False, False),   # four-row units, no ReLU
    (5, 32, 32, 64, 64, True, True),      # one image of the last group of four, upsampled store
    (90, 32, 32, 192, 64, False, True),   # four-row units, weights streamed (six channel blocks)
    (2, 8, 128, 32, 64, False, True),     # one image per group, rows of 128
    (1, 6, 128, 128, 32, False, True),    # a height no taller unit divides, weights streamed
])
def test_rows_match_64_bit_sums(un, T, H, W, cin, cout, up, relu):
    g = torch.Generator(device="cuda").manual_seed(T + H + W + cin + cout)
    x = torch.rand((T, H, W, cin), generator=g, device="cuda").to(torch.bfloat16)
    wk = (torch.randn((cout, 9 * cin), generator=g, device="cuda") * (2.0 / (9 * cin)) ** 0.5).to(torch.bfloat16)
    b = torch.randn((cout,), generator=g, device="cuda") * 0.05
    f, cy, coff = 2 if up else 1, cout + 32, 32
    y = torch.full((T, f * H, f * W, cy), 7.0, dtype=torch.bfloat16, device="cuda")
    un.conv3x3(x, wk, b, y, y_coff=coff, upsample=up, relu=relu)
    assert un.status() == 0
    assert torch.all(y[..., :coff] == 7.0)  # channels outside the layer's are untouched
    w = wk.double().view(cout, 3, 3, cin).permute(0, 1, 2, 3)
    z = _conv64(x.double(), w) + b.double()
    absum = _conv64(x.double().abs(), w.abs())
    o = torch.relu(z) if relu else z
    if up:
        o, absum = (a.repeat_interleave(2, 1).repeat_interleave(2, 2) for a in (o, absum))
    got = y[..., coff:].double()
    big = torch.maximum(o.abs(), got.abs()).clamp(min=2.0 ** -126)
    half_step = torch.exp2(torch.floor(torch.log2(big)) - 8)
    tol = 2 * 9 * cin * U * absum * (1 + 2.0 ** -7) + 2.0 ** -23 * big + half_step
    bad = (got - o).abs() > tol
    assert not bad.any(), f"{int(bad.sum())} of {bad.numel()} outside the bound"


def test_colors_and_pools_do_not_depend_on_the_tile_count(un):
    """The network's colors (output layer and pools in the row form's epilogue) of 39 tiles at
    once, eight-row units, are bit for bit those of the same tiles alone and a few at a time
    (two-row units, half-empty image groups)."""
    from paper_2506_15183_gb300 import weights as W

    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.zeros((39, 64, 64, 32), dtype=torch.bfloat16, device="cuda")
    x[..., :6] = torch.rand((39, 64, 64, 6), generator=g, device="cuda")
    net = un.Inpainter(W.load_flat(), max_tiles=39)
    every = torch.empty((39, 64, 64, 3), device="cuda")
    net.forward(x, every)
    t0 = 0
    for n in (1, 3, 10, 25):
        some = torch.empty((n, 64, 64, 3), device="cuda")
        net.forward(x[t0:t0 + n].contiguous(), some)
        assert torch.equal(some, every[t0:t0 + n])
        t0 += n
    assert un.status() == 0
    net.close()
