"""The work a user of this library has it do, as cases that can be timed and compared.

A case names one entry point of the public API (``kind``) and its sizes; ``prepare`` makes
what a program holds before the call (seeded inputs, handles, weights), ``run`` is one
pass.  Frames are the seeded ray-cast scenes of ``scene`` at the sizes of its workloads
(256x256, the batch's four per-eye resolutions) and ragged ones; network inputs are seeded
tiles with the network's value ranges; the inpainter's weights are the committed ones.

kinds
  frame    ``Synthesizer`` on one frame (a headset's next frame; kernel_rows / nearest_first
           are the Patcher variants)
  imb      the same through the row-downsampled intermediate buffer
  pose     the same for a rotated and offset second eye
  host     ``yoro_synthesize_host``: frames that live in pinned host memory
  batch    ``yoro_synthesize_batch``: frames of several headsets in one launch
  inpaint  ``yoro_synthesize_zt`` and the learned inpainter on its holes (several frames:
           ``inpaint_batch``)
  conv     ``conv3x3``: one layer of the inpainter's network
  forward  the inpainter's network on prepared tiles
  train    training steps of the inpainter and the reading of loss and gradients
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_15183_gb300 as yoro
from paper_2506_15183_gb300 import scene
from paper_2506_15183_gb300 import unet as un
from paper_2506_15183_gb300 import weights as W

NEAR, FAR = 0.05, 1000.0
YAW, PITCH = 0.02, 0.01  # rad: the rotation of the second eye in the pose cases
EYE = (0.063, 0.005, 0.0)

# The network's 3x3 layers: side, input channels (padded to 32), output channels, channel
# stride and offset of the output buffer, upsampled store.
LAYERS = {
    "enc0a": (64, 32, 32, 32, 0, False), "enc0b": (64, 32, 32, 96, 0, False),
    "enc1a": (32, 32, 64, 64, 0, False), "enc1b": (32, 64, 64, 192, 0, False),
    "enc2a": (16, 64, 128, 128, 0, False), "enc2b": (16, 128, 128, 384, 0, False),
    "enc3a": (8, 128, 256, 256, 0, False), "enc3b": (8, 256, 256, 384, 128, True),
    "dec2a": (16, 384, 128, 128, 0, False), "dec2b": (16, 128, 128, 192, 64, True),
    "dec1a": (32, 192, 64, 64, 0, False), "dec1b": (32, 64, 64, 96, 32, True),
    "dec0a": (64, 96, 32, 32, 0, False), "dec0b": (64, 32, 32, 32, 0, False),
}
HOLE_CELLS = 0.43  # share of a headset frame's 64x64 cells that hold a hole (0.40-0.48 on its scenes)


def listed():
    return [
        # the smallest frame of the workloads: latency and launches count
        dict(name="frame_256x256", kind="frame", w=256, h=256, prims=16, ground=False),
        # a headset's per-eye frame, one at a time
        dict(name="frame_1832x1920", kind="frame", w=1832, h=1920, prims=200, ground=True),
        # a ragged frame: rows are not 16-byte aligned, the last words are partial
        dict(name="frame_1439x1601", kind="frame", w=1439, h=1601, prims=200, ground=True),
        # the same frame in pinned host memory: copies in, the kernel, copies out
        dict(name="host_1832x1920", kind="host", w=1832, h=1920, prims=200, ground=True),
        # a server's batch: four headsets of each of the four per-eye sizes in one launch
        dict(name="batch_16", kind="batch", n=16),
        # the paper's downsampled intermediate buffer with interpolation
        dict(name="imb4_1832x1920", kind="imb", w=1832, h=1920, prims=200, ground=True, div=4, interp=True),
        # a second eye that is rotated and offset: pixels leave their rows
        dict(name="pose_1832x1920", kind="pose", w=1832, h=1920, prims=200, ground=True),
        # one layer of the network, the widest of its full-resolution level
        dict(name="conv_dec0a_128", kind="conv", layer="dec0a", T=128),
        # the network on a few tiles: a small frame's holes, launches and latency
        dict(name="forward_8", kind="forward", T=8),
        # the network on every tile of a headset frame
        dict(name="forward_870", kind="forward", T=870),
        # a headset frame with learned inpainting
        dict(name="inpaint_1832x1920", kind="inpaint", frames=1, w=1832, h=1920, prims=200),
        # training at the batch size of the committed weights
        dict(name="train_64x4", kind="train", T=64, steps=4),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """Width and height in [lo, hi], together no more pixels than 2064 x 2208; any remainder."""
    w, h = _logint(rng, lo, hi), _logint(rng, lo, hi)
    return w, min(h, 2064 * 2208 // w)


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "imb", "pose", "host", "batch", "inpaint", "conv", "conv", "forward",
                       "train"])
    if kind in ("frame", "imb", "pose", "host"):
        w, h = _size(rng, 100, 2600)
        c = dict(kind=kind, w=w, h=h, prims=rng.randint(16, 300), ground=rng.random() < 0.8)
        if kind == "frame" and rng.random() < 0.25:
            c.update(kernel_rows=rng.choice([1, 5, 7]), nearest_first=rng.random() < 0.5)
        if kind == "imb":
            c.update(div=rng.choice([2, 4, 8, 16]), interp=rng.random() < 0.7)
        return c
    if kind == "batch":
        return dict(kind=kind, n=_logint(rng, 2, 16))
    if kind == "inpaint":
        w, h = _size(rng, 128, 2208)
        return dict(kind=kind, frames=rng.randint(1, 3), w=w, h=h, prims=rng.randint(50, 300))
    if kind == "conv":
        return dict(kind=kind, layer=rng.choice(sorted(LAYERS)), T=2 * _logint(rng, 1, 200))
    if kind == "forward":
        return dict(kind=kind, T=_logint(rng, 1, 600))
    return dict(kind="train", T=2 * _logint(rng, 2, 32), steps=rng.randint(1, 4))


# ---- inputs


def _scene(w, h, prims, ground=True, ipd=0.063):
    return scene.SceneConfig(w=w, h=h, n_prims=prims, ground=ground, log_depth=ground, zmin=0.1 if ground else 0.3,
                             zmax=100.0 if ground else 20.0, ipd=ipd, near=NEAR, far=FAR)


def _frame(cfg, seed):
    c, d, _ = scene.render(cfg, seed)
    return torch.from_numpy(c), torch.from_numpy(d)


def _field(g, n, c, cells):
    """Smooth random fields in [0, 1]: (n, c, 64, 64)."""
    low = torch.rand((n, c, cells, cells), generator=g, device="cuda")
    return torch.nn.functional.interpolate(low, size=(64, 64), mode="bilinear", align_corners=True)


def _tiles(n, seed):
    """n network inputs (64, 64, 32) as prepared tiles hold them (colors / 255, the hole
    mask, near / warped depth with zero at holes, near / source depth, 26 zero channels),
    their hole masks and a ground truth."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    color = (_field(g, n, 3, 9) + 0.1 * torch.rand((n, 3, 64, 64), generator=g, device="cuda")).clamp(0, 1)
    color = torch.round(color * 255) / 255
    hole = _field(g, n, 1, 7) > 0.68
    z = torch.exp(math.log(0.3) + _field(g, n, 2, 6) * math.log(100 / 0.3))
    x = torch.zeros((n, 64, 64, 32), dtype=torch.bfloat16, device="cuda")
    x[..., 0:3] = color.permute(0, 2, 3, 1)
    x[..., 3] = hole[:, 0]
    x[..., 4] = torch.where(hole[:, 0], torch.zeros_like(z[:, 0]), NEAR / z[:, 0])
    x[..., 5] = NEAR / z[:, 1]
    gt = (color + 0.1 * (torch.rand((n, 3, 64, 64), generator=g, device="cuda") - 0.5)).clamp(0, 1)
    gt = torch.round(gt * 255).to(torch.uint8).permute(0, 2, 3, 1).contiguous()
    return x, hole[:, 0].to(torch.uint8).contiguous(), gt


def _rotation():
    cy, sy, cp, sp = math.cos(YAW), math.sin(YAW), math.cos(PITCH), math.sin(PITCH)
    return [[cy, 0.0, -sy], [-sp * sy, cp, -sp * cy], [cp * sy, sp, cp * cy]]


class _State:
    def __init__(self, case):
        self.kind, self.case = case["kind"], case


def prepare(case, seed):
    s = _State(case)
    kind = s.kind
    if kind in ("frame", "imb", "pose", "host"):
        cfg = _scene(case["w"], case["h"], case["prims"], case["ground"])
        color, depth = _frame(cfg, seed)
        more = {}
        if kind == "imb":
            more = dict(imbuffer_div=case["div"], interpolate=case["interp"])
        elif kind == "pose":
            more = dict(pose=(_rotation(), EYE))
        elif kind == "frame":
            more = dict(kernel_rows=case.get("kernel_rows", 3), nearest_first=case.get("nearest_first", False))
        s.syn = yoro.Synthesizer(**cfg.camera(), **more)
        if kind == "host":
            s.color, s.depth = color.pin_memory(), depth.pin_memory()
            s.out = torch.empty((cfg.h, cfg.w, 4), dtype=torch.uint8, pin_memory=True)
            s.mask = torch.empty((cfg.h, cfg.w), dtype=torch.uint8, pin_memory=True)
        else:
            s.color, s.depth = color.cuda(), depth.cuda()
    elif kind == "batch":
        rng = np.random.default_rng(seed)
        s.frames = []
        for i in range(case["n"]):
            w, h = scene.BATCH_SIZES[i % len(scene.BATCH_SIZES)]
            cfg = _scene(w, h, int(rng.integers(50, 301)), ipd=float(np.float32(rng.uniform(0.055, 0.072))))
            color, depth = _frame(cfg, 64 * seed + i)
            s.frames.append(dict(cfg.camera(), color=color.cuda(), depth=depth.cuda(),
                                 out_color=torch.empty((h, w, 4), dtype=torch.uint8, device="cuda"),
                                 out_mask=torch.empty((h, w), dtype=torch.uint8, device="cuda")))
    elif kind == "inpaint":
        cfg = _scene(case["w"], case["h"], case["prims"])
        w, h = cfg.w, cfg.h
        s.handle = yoro.Synthesizer(**cfg.camera())
        s.net = un.Inpainter(W.load_flat(), max_w=w, max_h=h)
        s.frames = []
        for i in range(case["frames"]):
            color, depth = _frame(cfg, 8 * seed + i)
            s.frames.append((color.cuda(), depth.cuda(), torch.empty((h, w, 4), dtype=torch.uint8, device="cuda"),
                             torch.empty((h, w), dtype=torch.uint8, device="cuda"),
                             torch.empty((h, w), dtype=torch.float32, device="cuda")))
    elif kind == "conv":
        side, cin, cout, cstride, coff, up = LAYERS[case["layer"]]
        g = torch.Generator(device="cuda").manual_seed(seed)
        T, f = case["T"], 2 if up else 1
        s.x = torch.randn((T, side, side, cin), generator=g, device="cuda").clamp(min=0).to(torch.bfloat16)
        s.wk = (torch.randn((cout, 9 * cin), generator=g, device="cuda") * math.sqrt(2 / (9 * cin))).to(torch.bfloat16)
        s.bias = torch.randn((cout,), generator=g, device="cuda") * 0.05
        s.y = torch.zeros((T, f * side, f * side, cstride), dtype=torch.bfloat16, device="cuda")
    elif kind == "forward":
        s.x, _, _ = _tiles(case["T"], seed)
        s.rgb = torch.empty((case["T"], 64, 64, 3), dtype=torch.float32, device="cuda")
        s.net = un.Inpainter(W.load_flat(), max_tiles=case["T"])
    else:
        # The step size is far below the weights' rounding unit: every step does all of its
        # work (Adam and the rebuilding of the layers' weights too), and passes repeat.
        s.trainer = un.Trainer(W.init_params(seed), batch_tiles=case["T"], lr=1e-30)
        s.batches = [_tiles(case["T"], 16 * seed + i) for i in range(case["steps"])]
    return s


def run(s):
    if s.kind in ("frame", "imb", "pose"):
        out, mask = s.syn(s.color, s.depth)
        return {"out": out, "mask": mask}
    if s.kind == "host":
        yoro.yoro_synthesize_host(s.syn.handle, s.color, s.depth, s.out, s.mask)
        return {"out": s.out, "mask": s.mask}
    if s.kind == "batch":
        yoro.yoro_synthesize_batch(s.frames)
        return [(f["out_color"], f["out_mask"]) for f in s.frames]
    if s.kind == "inpaint":
        for color, depth, out, mask, zt in s.frames:
            yoro.yoro_synthesize_zt(s.handle.handle, color, depth, out, mask, zt)
        if len(s.frames) == 1:
            color, depth, out, mask, zt = s.frames[0]
            s.net.inpaint(out, mask, zt, depth, NEAR)
        else:
            s.net.inpaint_batch([(out, mask, zt, depth, NEAR) for color, depth, out, mask, zt in s.frames])
        return [(out, mask, zt) for color, depth, out, mask, zt in s.frames]
    if s.kind == "conv":
        _, _, _, _, coff, up = LAYERS[s.case["layer"]]
        un.conv3x3(s.x, s.wk, s.bias, s.y, y_coff=coff, upsample=up)
        return s.y
    if s.kind == "forward":
        s.net.forward(s.x, s.rgb)
        return s.rgb
    for x, hole, gt in s.batches:
        s.trainer.step(x, gt, hole)
    return {"loss": s.trainer.read("loss"), "grads": s.trainer.read("grads")}


def work(case):
    kind = case["kind"]
    if kind in ("frame", "imb", "pose", "host"):  # 8 B in, 5 B out per pixel (the cells' depths alone with the buffer)
        depth = 4 / case["div"] if kind == "imb" else 4
        return {"bytes": case["w"] * case["h"] * (9 + depth), "flops": 0}
    if kind == "batch":
        sizes = [scene.BATCH_SIZES[i % len(scene.BATCH_SIZES)] for i in range(case["n"])]
        return {"bytes": sum(13 * w * h for w, h in sizes), "flops": 0}
    per_tile = W.flops_per_tile()
    params = 4 * W.count()
    if kind == "inpaint":
        w, h = case["w"], case["h"]
        cells = math.ceil(w / 64) * math.ceil(h / 64) * HOLE_CELLS
        return {"bytes": case["frames"] * 17 * w * h + params, "flops": case["frames"] * cells * per_tile}
    if kind == "conv":
        side, cin, cout, _, _, up = LAYERS[case["layer"]]
        px = case["T"] * side * side
        return {"bytes": px * 2 * (cin + (4 if up else 1) * cout) + 18 * cin * cout, "flops": px * 18 * cin * cout}
    if kind == "forward":  # 6 channels of 2 bytes in, 3 floats out
        return {"bytes": case["T"] * 4096 * (12 + 12) + params, "flops": case["T"] * per_tile}
    # per step: inputs, Adam's three arrays read and written; forward and two products backward
    return {"bytes": case["steps"] * (case["T"] * 4096 * (12 + 4) + 7 * params),
            "flops": case["steps"] * 3 * case["T"] * per_tile}


# ---- the computed numbers in 64 bits


def _r(t):
    """Rounded to bfloat16, in 64 bits."""
    return t.to(torch.bfloat16).double()


def _conv64(x, w):
    """x (T, H, W, Cin), w (Cout, Cin, 3, 3) -> (T, H, W, Cout), zero padding."""
    T, H, Wd, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    y = 0
    for dy in range(3):
        for dx in range(3):
            y = y + xp[:, dy:dy + H, dx:dx + Wd] @ w[:, :, dy, dx].t()
    return y


def _up(a):
    return a.repeat_interleave(2, 1).repeat_interleave(2, 2)


def _pool(a):
    T, H, Wd, C = a.shape
    return a.view(T, H // 2, 2, Wd // 2, 2, C).permute(0, 1, 3, 5, 2, 4).reshape(T, H // 2, Wd // 2, C, 4)


def _net64(x, p):
    """The network on x (T, 64, 64, 6) with bfloat16 weights and activations and 64-bit sums:
    the colors, and every layer's input and output."""
    seen = {}

    def layer(name, a):
        y = _r(torch.relu(_conv64(a, p[name + ".w"]) + p[name + ".b"]))
        seen[name] = (a, y)
        return y

    a, skips = x, []
    for lvl in range(4):
        if lvl:
            a = _pool(a).amax(-1)
        a = layer(f"enc{lvl}b", layer(f"enc{lvl}a", a))
        skips.append(a)
    for lvl in (2, 1, 0):
        a = layer(f"dec{lvl}b", layer(f"dec{lvl}a", torch.cat([skips[lvl], _up(a)], -1)))
    return torch.sigmoid(a @ p["out.w"].t() + p["out.b"]), a, seen


def _params64(flat):
    d = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in W.split(flat).items()}
    return {k: _r(v) if k.endswith(".w") else v.double() for k, v in d.items()}


def _grads64(x, hole, gt, p):
    """Loss and the gradient as one array in the parameters' order (bfloat16 activations and
    layer gradients, 64-bit sums)."""
    s, last, seen = _net64(x, p)
    m = hole.double()[..., None]
    n = 3 * float(m.sum())
    err = (s - gt.double() / 255) * m
    dz = 2 * err / n * s * (1 - s)
    grads = {"out.w": torch.einsum("thwk,thwc->kc", dz, last), "out.b": dz.sum((0, 1, 2))}

    def back(name, dy):
        a, y = seen[name]
        H, Wd = y.shape[1:3]
        d = torch.where(y > 0, dy, torch.zeros_like(dy))
        grads[name + ".b"] = d.sum((0, 1, 2))
        d = _r(d)
        ap = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1)).reshape(a.shape[0], H + 2, Wd + 2, -1)
        flat_d = d.reshape(-1, d.shape[-1])
        w = p[name + ".w"]
        gw = torch.empty_like(w)
        for ky in range(3):
            for kx in range(3):
                gw[:, :, ky, kx] = flat_d.t() @ ap[:, ky:ky + H, kx:kx + Wd].reshape(flat_d.shape[0], -1)
        grads[name + ".w"] = gw
        if name == "enc0a":
            return None
        return _r(_conv64(d, w.flip(2, 3).transpose(0, 1)))

    g = dz @ p["out.w"]
    skip = {}
    for lvl in (0, 1, 2):
        d = back(f"dec{lvl}a", back(f"dec{lvl}b", g))
        c = W.WIDTHS[lvl]
        skip[lvl], d = d[..., :c], d[..., c:]
        T, H, Wd, C = d.shape
        g = d.view(T, H // 2, 2, Wd // 2, 2, C).sum((2, 4))
    for lvl in (3, 2, 1, 0):
        d = back(f"enc{lvl}a", back(f"enc{lvl}b", g if lvl == 3 else g + skip[lvl]))
        if lvl:  # to the first maximum of each window
            win = _pool(seen[f"enc{lvl - 1}b"][1])
            first = torch.zeros_like(win).scatter_(-1, win.argmax(-1, keepdim=True), 1.0)
            T, h2, w2, C = d.shape
            g = (first * d[..., None]).view(T, h2, w2, C, 2, 2).permute(0, 1, 4, 2, 5, 3).reshape(T, 2 * h2, 2 * w2, C)
    out = []
    for name, _, _ in W.layers():
        out += [grads[name + ".w"].reshape(-1), grads[name + ".b"]]
    return float((err * err).sum() / n), torch.cat(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "conv":
        s = prepare(case, seed)
        side, cin, cout, cstride, coff, up = LAYERS[case["layer"]]
        w = s.wk.double().view(cout, 3, 3, cin).permute(0, 3, 1, 2)
        y = s.y.double()
        for t in range(0, case["T"], 16):
            z = torch.relu(_conv64(s.x[t:t + 16].double(), w) + s.bias.double())
            y[t:t + 16, ..., coff:coff + cout] = _up(z) if up else z
        return y
    if kind == "forward":
        x, _, _ = _tiles(case["T"], seed)
        p = _params64(W.load_flat())
        return torch.cat([_net64(x[t:t + 32, ..., :6].double(), p)[0] for t in range(0, case["T"], 32)])
    if kind == "train":
        x, hole, gt = _tiles(case["T"], 16 * seed + case["steps"] - 1)
        loss, grads = _grads64(x[..., :6].double(), hole, gt, _params64(W.init_params(seed)))
        return {"loss": np.array([loss]), "grads": grads}
    return None  # whole numbers: the frames' bytes
