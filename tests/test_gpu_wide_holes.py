"""General poses and the intermediate buffer where their band kernels change course, byte for
byte against the oracle (needs a GPU): holes hundreds of columns wide beside wide occluders
(kernels whose words are passed over by their largest depth), the scatter's two ways to divide, and frames
whose bands take several waves (band heights below the tallest)."""
import math

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


def _occluders(w, h, seed):
    """A far, smooth background behind a few wide near slabs: wide holes, and kernels full of
    foreground candidates."""
    rng = np.random.default_rng(seed)
    depth = np.full((h, w), 40.0, np.float32) + rng.uniform(0, 1, (h, w)).astype(np.float32)
    for _ in range(6):
        x0, y0 = int(rng.integers(0, w)), int(rng.integers(0, h))
        depth[y0:y0 + int(rng.integers(2, h // 2 + 3)), x0:x0 + int(rng.integers(1, w // 2 + 2))] = \
            np.float32(rng.uniform(0.3, 3.0))
    color = rng.integers(0, 256, (h, w, 4)).astype(np.uint8)
    return color, depth


def _rot(yaw, pitch):
    cy, sy, cp, sp = math.cos(yaw), math.sin(yaw), math.cos(pitch), math.sin(pitch)
    return [[cy, 0.0, -sy], [-sp * sy, cp, -sp * cy], [cp * sy, sp, cp * cy]]


@pytest.mark.parametrize("w,h,fx,near,rows", [
    (700, 90, 333.3, 0.05, 3), (1031, 64, 515.5, 0.05, 3), (1031, 64, 515.5, 1e-12, 3), (500, 70, 250.0, 0.05, 5),
    (1832, 420, 916.0, 0.05, 3), (257, 5, 77.7, 0.05, 1)])
@pytest.mark.parametrize("yaw,pitch,c", [(0.02, 0.01, (0.063, 0.005, 0.0)), (-0.05, 0.0, (0.6, -0.2, 0.1)),
                                          (0.0, 0.0, (1.1, 0.0, 0.0))])
def test_pose_bytes(yoro, w, h, fx, near, rows, yaw, pitch, c):
    import oracle

    color, depth = _occluders(w, h, w + h + rows)
    rot = _rot(yaw, pitch)
    syn = yoro.Synthesizer(w, h, fx, fx * 1.01, w / 2 + 0.25, h / 2, 0.0, near=near, far=1000.0, kernel_rows=rows,
                           pose=(rot, c))
    out, mask = syn(torch.from_numpy(color).cuda(), torch.from_numpy(depth).cuda())
    ref, rmask = oracle.synthesize_pose(color, depth, np.float32(fx), np.float32(fx * 1.01), np.float32(w / 2 + 0.25),
                                        np.float32(h / 2), np.array(rot, np.float32), np.array(c, np.float32),
                                        np.float32(near), np.float32(1000.0), kernel_rows=rows)
    assert np.array_equal(mask.cpu().numpy(), rmask)
    assert np.array_equal(out.cpu().numpy(), ref)
    syn.close()


@pytest.mark.parametrize("rot,c", [
    (np.eye(3), (-3e38, 0.0, -1e38)),                     # p'.z = 1e38: its reciprocal is a subnormal number
    (np.diag([1e38, 1.0, 1e38]), (-2.5, 0.0, -1.0)),      # the same by the rotation
    (np.eye(3) * 9e8, (0.063, 0.0, 0.0))])                # just inside the range of the estimates
def test_pose_bytes_far_out_of_scale(yoro, rot, c):
    """Rotations and positions are free as long as they are finite: where 1 / p'.z underflows the
    targets come from the divisions themselves."""
    import oracle

    w, h, one = 48, 20, np.float32(1.0)
    color, depth = _occluders(w, h, 5)
    depth = (depth * 0.001).astype(np.float32)
    rot, c = np.array(rot, np.float32), np.array(c, np.float32)
    syn = yoro.Synthesizer(w, h, 1.0, 1.0, 16.5, 8.5, 0.0, near=1e-4, far=1000.0, pose=(rot, c))
    out, mask = syn(torch.from_numpy(color).cuda(), torch.from_numpy(depth).cuda())
    ref, rmask = oracle.synthesize_pose(color, depth, one, one, np.float32(16.5), np.float32(8.5), rot, c,
                                        np.float32(1e-4), np.float32(1000.0))
    assert np.array_equal(mask.cpu().numpy(), rmask)
    assert np.array_equal(out.cpu().numpy(), ref)
    syn.close()


@pytest.mark.parametrize("w,h,div,interp", [(3000, 640, 4, True), (3001, 640, 2, True), (2999, 500, 16, False),
                                            (1832, 330, 4, True)])
def test_imbuffer_bytes_over_several_waves(yoro, w, h, div, interp):
    import oracle

    color, depth = _occluders(w, h, w + div)
    syn = yoro.Synthesizer(w, h, w / 2, w / 2, w / 2, h / 2, 0.063, kernel_rows=3, imbuffer_div=div, interpolate=interp)
    out, mask = syn(torch.from_numpy(color).cuda(), torch.from_numpy(depth).cuda())
    ref, rmask = oracle.synthesize_imb(color, depth, np.float32(w / 2), np.float32(0.063), np.float32(0.05),
                                       np.float32(1000.0), div, interp)
    assert np.array_equal(mask.cpu().numpy(), rmask)
    assert np.array_equal(out.cpu().numpy(), ref)
    syn.close()


def test_wide_frame_over_several_waves(yoro):
    import oracle

    w, h = 5003, 470
    color, depth = _occluders(w, h, 3)
    syn = yoro.Synthesizer(w, h, w / 2, w / 2, w / 2, h / 2, 0.063)
    out, mask = syn(torch.from_numpy(color).cuda(), torch.from_numpy(depth).cuda())
    ref, rmask = oracle.synthesize(color, depth, w / 2, w / 2, w / 2, h / 2, 0.063, 0.05, 1000.0)
    assert np.array_equal(mask.cpu().numpy(), rmask)
    assert np.array_equal(out.cpu().numpy(), ref)
    syn.close()
