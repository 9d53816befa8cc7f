"""Benchmark: right-eye synthesis throughput at 1832x1920 on GB300.

One step = the whole path (disparity, nearest-wins warp, gather, hole edges, hole
fill) over one 1832x1920 frame through the C ABI (``yoro_synthesize``), inputs
already resident in HBM.  Frames rotate through a pool of distinct seeded scenes
whose inputs and outputs together exceed twice the L2 size, so every step reads
and writes HBM.  Prints one JSON line (rank 0).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl yoro|reference]

Multi-GPU: one process per GPU (torchrun); every rank synthesizes its own frames
(independent replicas, no collective on the data path; scaling "weak"), and the
value is the frames of all ranks over the slowest rank's time.

``--impl reference`` times the CPU oracle (the definition of the method, plain C; its
all-core build, OpenMP over rows) on the same workload; under torchrun only rank 0
runs it.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import re
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "2nd-eye Mpix/s and frames/s at 1832x1920 (% HBM peak); p50/p99 frame latency"
UNIT = "Mpix/s"
BYTES_PER_PIXEL = 13  # read 4 B depth + 4 B color, write 4 B color + 1 B mask
KERNEL = "fused_single"
CSRC = os.path.join(ROOT, "paper_2506_15183_gb300", "csrc")
PROFILE_TRAFFIC = os.path.join(ROOT, "profiles", "traffic.json")


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=20000)
    p.add_argument("--warmup", type=int, default=200)
    p.add_argument("--impl", choices=["yoro", "reference"], default="yoro")
    p.add_argument("--pool", type=int, default=0, help="frames in the rotating pool (0: auto, >= 8)")
    p.add_argument("--cpu-seconds", type=float, default=10.0, help="bounded CPU-oracle sample")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--no-e2e", action="store_true", help="skip the host-buffer leg (profiling runs)")
    p.add_argument("--serve-seconds", type=float, default=3.0, help="serve workload: paced run length")
    p.add_argument("--workload", choices=["quest", "batch", "serve", "imbuffer", "pose", "inpaint"], default="quest",
                   help="quest: one 1832x1920 frame per step (the headline); batch: the 64-frame mixed batch; "
                        "serve: 8 headset streams through the serving loop; imbuffer: the 1832x1920 frames "
                        "through the row-downsampled intermediate buffer; pose: the 1832x1920 frames for a "
                        "rotated, vertically offset second eye; inpaint: the learned inpainter (network on 64x64 "
                        "tiles and the frame path)")
    p.add_argument("--imbuffer-div", type=int, default=4, help="imbuffer workload: source pixels per cell")
    p.add_argument("--no-interpolate", action="store_true", help="imbuffer workload: no linear interpolation")
    p.add_argument("--no-tune", action="store_true", help="batch workload: skip the band-height autotuner")
    p.add_argument("--tiles", type=int, default=0,
                   help="inpaint workload: tiles per network step (0: every tile of a 1832x1920 frame, 870)")
    p.add_argument("--streams", type=int, default=4,
                   help="streams the steps are issued on, round-robin (frames overlap on the GPU)")
    return p.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def frame_seeds(rank: int, world: int, pool: int):
    """Seeds of the frames rank `rank` synthesizes: disjoint across ranks (independent
    replicas on different scenes), seeds 1..pool on rank 0."""
    return [1 + rank * pool + i for i in range(pool)]


def max_over_ranks(t_ms: float, world: int, device=None) -> float:
    """Slowest rank's timed-region duration (the whole-job time)."""
    if world <= 1:
        return t_ms
    import torch
    import torch.distributed as dist

    t = torch.tensor([t_ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def _code_only(src: str) -> str:
    """C/CUDA source without comments and blank space: what the compiler sees."""
    src = re.sub(r"/\*.*?\*/", " ", src, flags=re.S)
    src = re.sub(r"//[^\n]*", " ", src)
    return " ".join(src.split())


KERNEL_SOURCES = ("fused.cu", "yoro_device.cuh", "yoro_internal.h")  # what the fused kernel is built from


def csrc_digest() -> str:
    """Digest of the fused kernel's sources (comments and layout ignored), to tell
    whether stored ncu counters still describe the kernel."""
    h = hashlib.sha256()
    for name in KERNEL_SOURCES:
        h.update(_code_only(open(os.path.join(CSRC, name), encoding="utf-8").read()).encode())
    return h.hexdigest()[:16]


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        d = json.load(open(path))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def ncu_traffic():
    """Per-launch DRAM bytes of the timed kernel from the committed ncu summary, if it was
    taken on the current kernel sources; else None."""
    if not os.path.exists(PROFILE_TRAFFIC):
        return None
    d = json.load(open(PROFILE_TRAFFIC))
    if d.get("csrc_digest") != csrc_digest():
        return None
    return d.get("dram_bytes_per_launch")


class ClockSampler:
    """nvidia-smi clock/throttle samples while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.rows = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                self.rows.append(parts)

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.thread.join(timeout=5)
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"], "samples": 0}
        sm = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        smax = [float(r[2]) for r in self.rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({n for r in self.rows for n, v in zip(names, r[5:9]) if v.lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": reasons, "samples": len(self.rows)}


def make_pool(cfg, seeds, device):
    import torch

    from paper_2506_15183_gb300 import scene

    pool = []
    for seed in seeds:
        c, d, _ = scene.render(cfg, seed)
        pool.append(dict(color=torch.from_numpy(c).to(device), depth=torch.from_numpy(d).to(device),
                         out=torch.empty((cfg.h, cfg.w, 4), dtype=torch.uint8, device=device),
                         mask=torch.empty((cfg.h, cfg.w), dtype=torch.uint8, device=device),
                         host=(c, d)))
    return pool


def _time_oracle(cfg, frames, seconds, all_cores):
    import oracle

    n = 0
    t0 = time.perf_counter()
    while True:
        c, d = frames[n % len(frames)]
        oracle.synthesize(c, d, cfg.fx, cfg.fy, cfg.cx, cfg.cy, cfg.ipd, cfg.near, cfg.far, all_cores=all_cores)
        n += 1
        dt = time.perf_counter() - t0
        if dt >= seconds and n >= 3:
            break
    return n, dt


def cpu_baseline(cfg, frames, seconds):
    """The oracle as it stands on pool frames: the all-core build (the same C source
    with OpenMP over rows, every host core) for `seconds`, then the one-thread build
    for `seconds`.  `value` and `cores` are the all-core leg's."""
    import oracle

    cores = oracle.threads(all_cores=True)
    n_mt, dt_mt = _time_oracle(cfg, frames, seconds, True)
    n_1, dt_1 = _time_oracle(cfg, frames, seconds, False)
    return {"value": round(n_mt * cfg.w * cfg.h / dt_mt / 1e6, 3), "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"{n_mt} frames of the 1832x1920 workload (seeds 1-{min(n_mt, len(frames))}), {dt_mt:.1f} s "
                      f"on {cores} host threads (OpenMP over rows); one-thread build: {n_1} frames in {dt_1:.1f} s",
            "one_core": {"value": round(n_1 * cfg.w * cfg.h / dt_1 / 1e6, 3), "unit": UNIT, "cores": 1}}


def run_reference(args, rank, world, budget_s: float = 120.0):
    """The CPU oracle on the same workload.  Each step synthesizes a band of rows of a
    1832x1920 frame (plus one halo row above and below, not counted), the band height
    chosen from a one-frame calibration so that the warm-up and timed steps together
    take about `budget_s` seconds.  Value = output pixels / time."""
    from paper_2506_15183_gb300 import scene

    if rank != 0:
        return
    import oracle

    oracle.build()
    cfg = scene.quest_config()
    frames = [scene.render(cfg, 1 + i)[:2] for i in range(4)]

    cores = oracle.threads(all_cores=True)

    def run_band(i, rows):
        c, d = frames[i % len(frames)]
        y0 = (i * 97) % max(1, cfg.h - rows + 1)
        a, b = max(0, y0 - 1), min(cfg.h, y0 + rows + 1)
        oracle.synthesize(c[a:b], d[a:b], cfg.fx, cfg.fy, cfg.cx, cfg.cy, cfg.ipd, cfg.near, cfg.far,
                          all_cores=True)

    t0 = time.perf_counter()
    for i in range(len(frames)):
        run_band(i, cfg.h)
    t_frame = (time.perf_counter() - t0) / len(frames)
    per_step = budget_s / max(1, args.steps + args.warmup)
    rows = int(max(4, min(cfg.h, cfg.h * per_step / max(t_frame, 1e-6))))
    for i in range(args.warmup):
        run_band(i, rows)
    t0 = time.perf_counter()
    for i in range(args.steps):
        run_band(i, rows)
    dt = time.perf_counter() - t0
    mpix = args.steps * rows * cfg.w / dt / 1e6
    sample = (f"{args.steps} steps of {rows} rows x {cfg.w} px (+2 halo rows) of the 1832x1920 workload, "
              f"seeds 1-4, {cores} host threads (the oracle's all-core build: OpenMP over rows)")
    line = {
        "impl": "reference", "metric": METRIC, "value": round(mpix, 3), "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(1e3 * dt / args.steps, 3),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "quest 1832x1920: 200 primitives + ground plane, front depth log-uniform 0.1-100 m, "
                               "IPD 0.063 m, 90 deg HFOV", "w": cfg.w, "h": cfg.h, "rows_per_step": rows},
        "frames_per_s": round(args.steps * rows / cfg.h / dt, 3),
        "cpu_baseline": {"value": round(mpix, 3), "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": round(mpix, 3), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def run_batch(args):
    """The batched workload: 64 frames (16 each of 1024x1024, 1440x1600, 1832x1920 and
    2064x2208), each its own seeded scene, synthesized by one yoro_synthesize_batch launch
    per step.  Two copies of the batch alternate so that consecutive steps touch
    different memory (2 x 64 frames of inputs and outputs > 2x L2)."""
    import multiprocessing as mp
    from concurrent.futures import ProcessPoolExecutor

    import torch

    import paper_2506_15183_gb300 as yoro
    from paper_2506_15183_gb300 import scene

    specs = scene.batch_configs(64)
    with ProcessPoolExecutor(max_workers=min(16, os.cpu_count() or 2), mp_context=mp.get_context("spawn")) as ex:
        data = list(ex.map(_render_left, specs))
    copies = []
    for _ in range(2):
        frames = []
        for (cfg, seed), (c, d) in zip(specs, data):
            frames.append(dict(cfg.camera(), color=torch.from_numpy(c).cuda(), depth=torch.from_numpy(d).cuda(),
                               out_color=torch.empty((cfg.h, cfg.w, 4), dtype=torch.uint8, device="cuda"),
                               out_mask=torch.empty((cfg.h, cfg.w), dtype=torch.uint8, device="cuda")))
        copies.append(frames)
    npx = sum(cfg.w * cfg.h for cfg, _ in specs)
    stream = torch.cuda.Stream()
    wmax = max(cfg.w for cfg, _ in specs)
    yoro.yoro_reset_tuning()
    band_default = yoro.yoro_batch_band(wmax)
    band = band_default if args.no_tune else yoro.yoro_tune_batch(copies[0], reps=3, stream=stream)
    for i in range(args.warmup):
        yoro.yoro_synthesize_batch(copies[i % 2], stream=stream)
    torch.cuda.synchronize()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for i in range(args.steps):
        yoro.yoro_synthesize_batch(copies[i % 2], stream=stream)
    ev1.record(stream)
    stream.synchronize()
    t_ms = ev0.elapsed_time(ev1)
    secs = t_ms / 1e3
    peak, _ = measured_peaks()
    achieved = BYTES_PER_PIXEL * npx * args.steps / secs / 1e9
    print(json.dumps({
        "metric": "2nd-eye Mpix/s, batched workload (64 mixed frames per launch)", "value": round(npx * args.steps / secs / 1e6, 3),
        "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(t_ms / args.steps, 4),
        "higher_is_better": True, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "batch: 16 each of 1024x1024, 1440x1600, 1832x1920, 2064x2208; 50-300 primitives; "
                               "IPD U(0.055, 0.072) m; seeds 1000-1063", "frames_per_step": 64, "pixels_per_step": npx,
                   "entry_point": "yoro_synthesize_batch", "band_rows": band, "band_rows_untuned": band_default,
                   "tuned": not args.no_tune},
        "frames_per_s": round(64 * args.steps / secs, 1),
        "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                     "frac": round(achieved / peak, 4)},
    }), flush=True)


# second-eye pose of the pose workload: yaw 0.02 rad, pitch 0.01 rad, at (0.063, 0.005, 0) m
POSE_YAW, POSE_PITCH, POSE_POS = 0.02, 0.01, (0.063, 0.005, 0.0)


def _pose_rotation():
    cy, sy = np.cos(POSE_YAW), np.sin(POSE_YAW)
    cp, sp = np.cos(POSE_PITCH), np.sin(POSE_PITCH)
    ry = np.array([[cy, 0, sy], [0, 1, 0], [-sy, 0, cy]])
    rx = np.array([[1, 0, 0], [0, cp, -sp], [0, sp, cp]])
    return (rx @ ry).astype(np.float32)


def run_variant(args):
    """The 1832x1920 workload through a variant path: the row-downsampled intermediate
    buffer (yoro_create_imb) or a general second-eye pose (yoro_create_pose).  The same
    rotating pool as the headline, one handle per stream (the paths may use handle-owned
    scratch), steps round-robin over the streams.  Algorithmic bytes per pixel: 4 color
    read (+ 4 / div depth for the buffer, + 4 depth for the pose), 4 color + 1 mask
    written."""
    import torch

    import paper_2506_15183_gb300 as yoro
    from paper_2506_15183_gb300 import scene

    cfg = scene.quest_config()
    npx = cfg.w * cfg.h
    pool = make_pool(cfg, frame_seeds(0, 1, max(8, args.pool)), "cuda")
    div, interp = args.imbuffer_div, not args.no_interpolate
    nstreams = max(1, args.streams)
    streams = [torch.cuda.Stream() for _ in range(nstreams)]
    cam = cfg.camera()
    if args.workload == "pose":
        handles = [yoro.yoro_create_pose(cam["w"], cam["h"], cam["fx"], cam["fy"], cam["cx"], cam["cy"],
                                         _pose_rotation(), POSE_POS, cam["near"], cam["far"]) for _ in streams]
    else:
        handles = [yoro.yoro_create_imb(**cam, imbuffer_div=div, interpolate=interp) for _ in streams]

    def step(i):
        f = pool[i % len(pool)]
        k = i % nstreams
        yoro.yoro_synthesize(handles[k], f["color"], f["depth"], f["out"], f["mask"], stream=streams[k])

    for i in range(args.warmup):
        step(i)
    torch.cuda.synchronize()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    ev0.record(streams[0])
    for st in streams[1:]:
        st.wait_event(ev0)
    for i in range(args.steps):
        step(i)
    for st in streams[1:]:
        done = torch.cuda.Event()
        done.record(st)
        streams[0].wait_event(done)
    ev1.record(streams[0])
    streams[0].synchronize()
    t_ms = ev0.elapsed_time(ev1)
    for k, hdl in enumerate(handles):
        status = yoro.yoro_stream_status(hdl, streams[k])
        if status != 0:
            raise yoro.YoroError(status, "kernel status")
        yoro.yoro_destroy(hdl)
    secs = t_ms / 1e3
    pose = args.workload == "pose"
    bpp = 4 + 4 + 4 + 1 if pose else 4 + 4 / div + 4 + 1
    peak, _ = measured_peaks()
    achieved = bpp * npx * args.steps / secs / 1e9
    config = ({"workload": "quest 1832x1920, second eye rotated (yaw 0.02, pitch 0.01 rad) at (0.063, 0.005, 0) m",
               "entry_point": "yoro_synthesize (yoro_create_pose handle)"} if pose else
              {"workload": "quest 1832x1920 through the intermediate buffer", "imbuffer_div": div,
               "interpolate": interp, "entry_point": "yoro_synthesize (yoro_create_imb handle)"})
    config.update(streams=nstreams, pool_frames=len(pool))
    print(json.dumps({
        "metric": "2nd-eye Mpix/s, " + ("general-pose variant" if pose else "intermediate-buffer variant"),
        "value": round(npx * args.steps / secs / 1e6, 3),
        "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(t_ms / args.steps, 5),
        "higher_is_better": True, "dtype": "f32", "data": "synthetic",
        "config": config,
        "frames_per_s": round(args.steps / secs, 1),
        "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                     "frac": round(achieved / peak, 4), "bytes_per_pixel": bpp},
        "gpu_launches": (3 if pose else 1) * args.steps,  # pose: scatter, gather, fill; buffer: one band kernel
    }), flush=True)


def _render_pose(spec):
    from paper_2506_15183_gb300 import scene

    cfg, seed, eye_x = spec
    c, d, _ = scene.render(cfg, seed, eye_x=eye_x, nthreads=2)
    return c, d


def run_serve(args):
    """The serving workload: 8 headset streams (1440x1600, 1832x1920, 2064x2208 at 72, 90
    and 120 Hz) through the library's serving loop (continuous batching, resident slots).
    Each stream's renderer is a pool of left eyes pre-rendered on the host along a seeded
    random walk of the head (8 poses per stream, 200-primitive scene); at every refresh
    it copies the next pose into a free slot of its stream and submits it.  Reports each
    stream's frames/s and submit-to-done latency p50/p99, then the saturation throughput
    with every stream resubmitting as soon as a slot frees up."""
    import multiprocessing as mp
    import time
    from concurrent.futures import ProcessPoolExecutor

    import numpy as np
    import torch

    import paper_2506_15183_gb300 as yoro
    from paper_2506_15183_gb300 import scene
    from paper_2506_15183_gb300.server import Server

    from paper_2506_15183_gb300 import unet as un
    from paper_2506_15183_gb300 import weights as W

    sizes = [(1440, 1600), (1832, 1920), (2064, 2208)]
    rates = [72.0, 90.0, 120.0]
    nstreams, poses, slots = 8, 32, 3
    rng = np.random.default_rng(2024)
    specs, streams = [], []
    for i in range(nstreams):
        w, h = sizes[i % 3]
        cfg = scene.quest_config().replace(w=w, h=h, ipd=float(rng.uniform(0.055, 0.072)))
        walk = np.cumsum(rng.normal(0.0, 0.004, poses))  # head x offset, metres
        streams.append(dict(cfg=cfg, hz=rates[i % 3]))
        specs += [(cfg, 5000 + i, float(x)) for x in walk]
    with ProcessPoolExecutor(max_workers=min(16, os.cpu_count() or 2), mp_context=mp.get_context("spawn")) as ex:
        data = list(ex.map(_render_pose, specs))
    for i, st in enumerate(streams):
        st["pool"] = [(torch.from_numpy(c).cuda(), torch.from_numpy(d).cuda()) for c, d in data[i * poses:(i + 1) * poses]]
    yoro.load_library()
    srv = Server(16 << 30, max_batch=64)
    params, weights_kind = (W.load_flat(), "trained") if W.exists() else (W.init_params(1), "initial")
    net = un.Inpainter(params, max_w=max(w for w, _ in sizes), max_h=max(h for _, h in sizes))
    copy_stream = torch.cuda.Stream()
    for i, st in enumerate(streams):
        st["learned"] = i % 2 == 1  # every other stream repaints its holes with the network
        st["id"] = srv.admit(**st["cfg"].camera(), slots=slots, learned=st["learned"])
        st["views"] = [srv.slot(st["id"], k) for k in range(slots)]

    def run(seconds, paced):
        for st in streams:
            st["free"] = list(range(slots))
            st["next"] = 0.0
            st["lat"] = []
            st["n"] = 0
            st["inpainted"] = 0
        t0 = time.perf_counter()
        submitted = completed = 0
        while True:
            now = time.perf_counter() - t0
            if now > seconds:
                break
            for r in srv.poll(4096):
                st = streams[r.stream]
                st["free"].append(r.slot)
                st["lat"].append((r.done_ns - r.submit_ns) / 1e6)
                st["inpainted"] += r.inpainted
                completed += 1
            for st in streams:
                if st["free"] and (not paced or now >= st["next"]):
                    k = st["free"].pop(0)
                    c, d = st["pool"][st["n"] % poses]
                    ci, di, _, _ = st["views"][k]
                    with torch.cuda.stream(copy_stream):
                        ci.copy_(c, non_blocking=True)
                        di.copy_(d, non_blocking=True)
                    copy_stream.synchronize()
                    srv.submit(st["id"], k, tag=st["n"])
                    st["n"] += 1
                    submitted += 1
                    st["next"] = st["next"] + 1.0 / st["hz"] if paced else now
            if paced:
                time.sleep(0.0002)
        srv.drain(60000)
        for r in srv.poll(1 << 16):
            streams[r.stream]["lat"].append((r.done_ns - r.submit_ns) / 1e6)
        return time.perf_counter() - t0

    def report(secs):
        out = []
        for st in streams:
            lat = sorted(st["lat"])
            out.append({"w": st["cfg"].w, "h": st["cfg"].h, "hz": st["hz"], "learned": st["learned"],
                        "frames": len(lat), "inpainted": st["inpainted"], "frames_per_s": round(len(lat) / secs, 1),
                        "latency_ms_p50": round(lat[len(lat) // 2], 3) if lat else None,
                        "latency_ms_p99": round(lat[int(0.99 * (len(lat) - 1))], 3) if lat else None})
        return out

    srv.set_inpainter(net)
    run(0.5, paced=True)  # warm-up
    secs = run(max(2.0, args.serve_seconds), paced=True)
    per_stream = report(secs)
    sat_secs = run(2.0, paced=False)
    sat_frames = sum(len(st["lat"]) for st in streams)
    sat_px = sum(len(st["lat"]) * st["cfg"].w * st["cfg"].h for st in streams)
    srv.drain(60000)
    # saturation again with the server's own feeder thread (no host loop in the way)
    for r in srv.poll(1 << 16):
        pass
    for st in streams:
        srv.feed(st["id"], st["pool"], nframes=1 << 40, hz=0.0)
    feed_n, feed_px = 0, 0
    t_f0 = time.perf_counter()
    while time.perf_counter() - t_f0 < 2.0:
        for r in srv.poll(1 << 16):
            st = streams[r.stream]
            feed_n += 1
            feed_px += st["cfg"].w * st["cfg"].h
        time.sleep(0.001)
    feed_secs = time.perf_counter() - t_f0
    srv.feed_stop()
    srv.drain(60000)
    srv.poll(1 << 16)
    srv.set_inpainter(None)  # the fallback: learned streams keep the paper's fill
    fb_secs = run(max(2.0, args.serve_seconds), paced=True)
    fallback = report(fb_secs)
    srv.close()
    net.close()
    print(json.dumps({
        "metric": "serving loop: 8 headset streams at their refresh rates (frames/s and submit-to-done latency)",
        "value": round(sum(p["frames_per_s"] for p in per_stream), 1), "unit": "frames/s", "n_gpus": 1,
        "higher_is_better": True, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "serve: 8 streams of 1440x1600, 1832x1920, 2064x2208 at 72/90/120 Hz; head x on a "
                               "seeded random walk, 32 poses per stream rendered on the host; 3 resident slots per "
                               "stream; streams 1, 3, 5, 7 with learned inpainting",
                   "entry_point": "yoro_server_submit (continuous batching)", "paced_seconds": round(secs, 2),
                   "inpainter_weights": weights_kind},
        "streams": per_stream,
        "fallback_streams": fallback,
        "saturation": {"frames_per_s": round(sat_frames / sat_secs, 1), "mpix_per_s": round(sat_px / sat_secs / 1e6, 1),
                       "what": "every stream resubmits as soon as one of its 3 slots frees up (host loop, one thread)"},
        "saturation_feeder": {"frames_per_s": round(feed_n / feed_secs, 1), "mpix_per_s": round(feed_px / feed_secs / 1e6, 1),
                              "what": "the same with the server's feeder thread copying pose frames into free slots "
                                      "(yoro_server_feed, no host loop); learned streams repainted"},
    }), flush=True)


def run_inpaint(args):
    """The learned inpainter: (1) the network alone on every 64x64 tile of a 1832x1920
    frame (870 tiles per step, inputs resident), timed with CUDA events, against the
    measured bfloat16 tensor peak; (2) the frame path: yoro_synthesize_zt then
    yoro_unet_inpaint on the quest frames (rotating pool), frames/s and per-frame latency."""
    import torch

    import paper_2506_15183_gb300 as yoro
    from paper_2506_15183_gb300 import scene
    from paper_2506_15183_gb300 import unet as un
    from paper_2506_15183_gb300 import weights as W

    cfg = scene.quest_config()
    if W.exists():
        params, weights_kind = W.load_flat(), "trained (paper_2506_15183_gb300/weights/unet.yw)"
    else:
        params, weights_kind = W.init_params(1), "initial (seeded He-normal)"
    ntx, nty = (cfg.w + 63) // 64, (cfg.h + 63) // 64
    T = args.tiles if args.tiles > 0 else ntx * nty
    net = un.Inpainter(params, max_tiles=T, max_w=cfg.w, max_h=cfg.h)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.zeros((T, 64, 64, 32), dtype=torch.bfloat16, device="cuda")
    x[..., :6] = torch.rand((T, 64, 64, 6), generator=g, device="cuda").to(torch.bfloat16)
    rgb = torch.empty((T, 64, 64, 3), dtype=torch.float32, device="cuda")
    stream = torch.cuda.Stream()
    for _ in range(max(3, args.warmup)):
        net.forward(x, rgb, stream=stream)
    stream.synchronize()
    steps = max(1, args.steps)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(steps):
        net.forward(x, rgb, stream=stream)
    ev1.record(stream)
    stream.synchronize()
    if un.status(stream) != 0:
        raise RuntimeError("inpainter kernel status")
    ms = ev0.elapsed_time(ev1) / steps
    flops = W.flops_per_tile() * T
    tflops = flops / (ms * 1e-3) / 1e12
    peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json"))) if os.path.exists(
        os.path.join(ROOT, "MEASURED_PEAKS.json")) else {}
    peak = float(peaks.get("bf16_tflops", 1900.0))
    # (2) the frame path on the quest pool
    pool = make_pool(cfg, frame_seeds(0, 1, 4), "cuda")
    hdl = yoro.yoro_create(**cfg.camera())
    zt = torch.empty((cfg.h, cfg.w), dtype=torch.float32, device="cuda")
    lat = []
    for i in range(max(3, args.warmup) + 20):
        f = pool[i % len(pool)]
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        yoro.yoro_synthesize_zt(hdl, f["color"], f["depth"], f["out"], f["mask"], zt, stream=stream)
        net.inpaint(f["out"], f["mask"], zt, f["depth"], cfg.near, stream=stream)
        b.record(stream)
        stream.synchronize()
        if i >= max(3, args.warmup):
            lat.append(a.elapsed_time(b))
    lat.sort()
    yoro.yoro_destroy(hdl)
    net.close()
    print(json.dumps({
        "metric": "learned inpainter: network TFLOP/s on 64x64 tiles; frame path ms (synthesis + inpainting)",
        "value": round(tflops, 2), "unit": "TFLOP/s", "n_gpus": 1, "steps": steps, "warmup": args.warmup,
        "ms_per_step": round(ms, 4), "higher_is_better": True, "dtype": "bf16 (fp32 accumulate)",
        "data": "synthetic", "weights": weights_kind,
        "config": {"workload": f"{T} 64x64 tiles per step ({ntx * nty}: every tile of a 1832x1920 frame), 4-level "
                               "U-Net 32/64/128/256", "flops_per_tile": W.flops_per_tile(), "tiles": T},
        "roofline": {"bound": "tensor", "achieved": round(tflops, 2), "peak": peak, "unit": "TFLOP/s",
                     "frac": round(tflops / peak, 4), "peak_source": "MEASURED_PEAKS.json bf16_tflops (burst)",
                     "traffic": None,
                     "traffic_note": "the network is 14 convolution launches and small kernels; DRAM bytes per "
                                     "convolution launch are in profiles/conv3x3_network.md"},
        "frame_path_ms": {"p50": round(lat[len(lat) // 2], 3), "p99": round(lat[int(0.99 * (len(lat) - 1))], 3),
                          "what": "yoro_synthesize_zt + yoro_unet_inpaint on one 1832x1920 frame (hole tiles only)"},
    }), flush=True)


def _render_left(spec):
    from paper_2506_15183_gb300 import scene

    cfg, seed = spec
    c, d, _ = scene.render(cfg, seed, nthreads=2)
    return c, d


def main():
    args = parse()
    rank, world, local = dist_env()
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    if args.workload == "batch":
        if rank == 0:
            run_batch(args)
        return
    if args.workload == "serve":
        if rank == 0:
            run_serve(args)
        return
    if args.workload in ("imbuffer", "pose"):
        if rank == 0:
            run_variant(args)
        return
    if args.workload == "inpaint":
        if rank == 0:
            run_inpaint(args)
        return

    import torch

    import paper_2506_15183_gb300 as yoro
    from paper_2506_15183_gb300 import scene

    if world > 1:
        import torch.distributed as dist

        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device(f"cuda:{local}"))
    device = torch.device(f"cuda:{local}")
    torch.cuda.set_device(device)
    lib = yoro.load_library()

    cfg = scene.quest_config()
    npx = cfg.w * cfg.h
    l2 = torch.cuda.get_device_properties(device).L2_cache_size
    pool_n = args.pool or max(8, int(np.ceil(2 * l2 / (BYTES_PER_PIXEL * npx))) + 1)
    pool = make_pool(cfg, frame_seeds(rank, world, pool_n), device)
    hdl = yoro.yoro_create(**cfg.camera())
    nstreams = max(1, args.streams)
    streams = [torch.cuda.Stream(device) for _ in range(nstreams)]
    stream = streams[0]
    calls = [[(hdl.ptr, f["color"].data_ptr(), f["depth"].data_ptr(), f["out"].data_ptr(), f["mask"].data_ptr(),
               st.cuda_stream) for f in pool] for st in streams]
    synth = lib.yoro_synthesize

    def step(i):
        return synth(*calls[i % nstreams][i % pool_n])

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    # the clock sampler starts first (nvidia-smi takes a moment to begin sampling), so that
    # the warm-up runs right before the timed region and the GPU does not idle between them
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    # warm-up
    for i in range(args.warmup):
        rc = step(i)
        if rc:
            raise yoro.YoroError(rc, "yoro_synthesize")
    torch.cuda.synchronize(device)

    # timed region: K back-to-back frames dealt round-robin over the streams
    barrier()
    torch.cuda.synchronize(device)
    # every stream waits for ev0 before its first step and ev1 waits for every stream, so
    # [ev0, ev1] spans all K steps; each wait is issued just before its stream's first step,
    # so the first frame is queued right after ev0
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    waiting = set(range(1, nstreams))
    for i in range(args.steps):
        k = i % nstreams
        if k in waiting:
            streams[k].wait_event(ev0)
            waiting.discard(k)
        step(i)
    for k in waiting:
        streams[k].wait_event(ev0)
    for st in streams[1:]:
        done = torch.cuda.Event()
        done.record(st)
        stream.wait_event(done)
    ev1.record(stream)
    stream.synchronize()
    barrier()
    torch.cuda.synchronize(device)
    clk = clocks.stop()
    t_ms = max_over_ranks(ev0.elapsed_time(ev1), world, device)
    status = yoro.yoro_stream_status(hdl, stream)
    if status != 0:
        raise yoro.YoroError(status, "kernel status")

    # per-frame device latency: one frame at a time, event pair around each launch
    lat = []
    n_lat = min(2000, max(200, args.steps // 10))
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n_lat)]
    for i, (a, b) in enumerate(evs):
        a.record(stream)
        synth(*calls[0][i % pool_n])
        b.record(stream)
    stream.synchronize()
    lat = sorted(a.elapsed_time(b) * 1e3 for a, b in evs)  # us

    # end-to-end through the host-buffer entry point: H2D inputs, kernel, D2H outputs per step
    e2e = None if args.no_e2e else run_e2e(yoro, lib, cfg, pool, device, steps=min(args.steps, 400), warmup=10)

    frames = args.steps * world
    secs = t_ms / 1e3
    mpix = frames * npx / secs / 1e6
    per_launch_s = secs / args.steps
    peak, peak_kind = measured_peaks()
    achieved = BYTES_PER_PIXEL * npx / per_launch_s / 1e9
    line = {
        "metric": METRIC, "value": round(mpix, 3), "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(t_ms / args.steps, 5), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "quest 1832x1920: 200 primitives + ground plane, front depth log-uniform 0.1-100 m, "
                               "IPD 0.063 m, 90 deg HFOV", "w": cfg.w, "h": cfg.h, "pool_frames": pool_n,
                   "l2_flush": f"rotating pool of {pool_n} frames ({pool_n * BYTES_PER_PIXEL * npx / 1e6:.0f} MB "
                               f"of inputs+outputs) > 2x L2 ({l2 / 1e6:.0f} MB)",
                   "parallelism": f"replicas{world}", "entry_point": "yoro_synthesize",
                   "streams": nstreams},
        "frames_per_s": round(frames / secs, 1),
        "hbm_frac_of_peak": round(achieved / peak, 4),
        "latency_us": {"p50": round(lat[len(lat) // 2], 2), "p99": round(lat[int(0.99 * (len(lat) - 1))], 2),
                       "what": "device time of one frame launched alone (CUDA events around one call)",
                       "samples": len(lat)},
        "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                     "what": "13 B per pixel x frames / timed region (launches overlap across streams)",
                     "frac": round(achieved / peak, 4), "traffic": ncu_traffic(),
                     "kernel": KERNEL, "bytes_per_launch": BYTES_PER_PIXEL * npx,
                     "peak_source": f"{peak_kind} (MEASURED_PEAKS.json hbm_gbs)" if peak_kind == "measured"
                     else "fallback 6.8 TB/s"},
        "e2e": e2e,
        "gpu_launches": args.steps,
        "clocks": clk,
    }
    if rank == 0 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(cfg, [f["host"] for f in pool], args.cpu_seconds)
    if rank == 0:
        print(json.dumps(line), flush=True)
    yoro.yoro_destroy(hdl)
    if world > 1:
        torch.distributed.destroy_process_group()


def run_e2e(yoro, lib, cfg, pool, device, steps, warmup):
    """Throughput through yoro_synthesize_host with pinned host buffers: each step copies
    its inputs host->device, synthesizes, and copies the right eye and mask back.  Three
    handles on three streams let copies of one frame overlap the kernel of another."""
    import torch

    npx = cfg.w * cfg.h
    nslot = 3
    hosts = []
    for i in range(nslot):
        c, d = pool[i % len(pool)]["host"]
        hosts.append((torch.from_numpy(c).pin_memory(), torch.from_numpy(d).pin_memory(),
                      torch.empty((cfg.h, cfg.w, 4), dtype=torch.uint8).pin_memory(),
                      torch.empty((cfg.h, cfg.w), dtype=torch.uint8).pin_memory()))
    streams = [torch.cuda.Stream(device) for _ in range(nslot)]
    handles = [yoro.yoro_create(**cfg.camera()) for _ in range(nslot)]
    calls = [(handles[i].ptr, *[t.data_ptr() for t in hosts[i]], streams[i].cuda_stream) for i in range(nslot)]
    fn = lib.yoro_synthesize_host
    for i in range(warmup):
        fn(*calls[i % nslot])
    torch.cuda.synchronize(device)
    t0 = time.perf_counter()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev0.record(streams[0])
    waiting = set(range(1, nslot))  # each stream waits for ev0 just before its first step
    for i in range(steps):
        if i % nslot in waiting:
            streams[i % nslot].wait_event(ev0)
            waiting.discard(i % nslot)
        rc = fn(*calls[i % nslot])
        if rc:
            raise yoro.YoroError(rc, "yoro_synthesize_host")
    for k in waiting:
        streams[k].wait_event(ev0)
    ends = []
    for s in streams:
        e = torch.cuda.Event(enable_timing=True)
        e.record(s)
        ends.append(e)
    torch.cuda.synchronize(device)
    wall = time.perf_counter() - t0
    t_ms = max(ev0.elapsed_time(e) for e in ends)
    for h in handles:
        yoro.yoro_destroy(h)
    return {"value": round(steps * npx / (t_ms / 1e3) / 1e6, 3), "unit": UNIT,
            "h2d_bytes_per_step": 8 * npx, "d2h_bytes_per_step": 5 * npx,
            "steps": steps, "wall_s": round(wall, 4), "entry_point": "yoro_synthesize_host (pinned host buffers)"}


if __name__ == "__main__":
    main()
