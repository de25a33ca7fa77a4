"""gs_map_add's means and log-scales are the FP64 values rounded to FP32, whatever the camera:
frames of pixels, and cameras and images outside the range of the FP32 pairs that carry most of
the arithmetic."""
import numpy as np
import pytest
import torch

from paper_2408_05635_gb300 import gs, scenes

pytestmark = pytest.mark.gpu


def _add(cam, pose, depth):
    m = gs.Map(max(int((depth > 0).sum()), 4), "cuda")
    m.add_from_frame(cam, torch.tensor(pose, dtype=torch.float64, device="cuda"),
                     torch.zeros(3, *depth.shape, device="cuda"), torch.tensor(depth, device="cuda"))
    n = m.n
    return m.p["means"][:n].cpu().numpy(), m.p["log_scales"][:n].cpu().numpy()


def _want(cam, pose, depth, dt=np.float64):
    """Means, the size of their terms, and log-scales."""
    v, u = [a.astype(dt) for a in np.nonzero(depth > 0)]
    d = depth[depth > 0].astype(dt)
    local = np.stack([(u - dt(cam.cx)) / dt(cam.fx) * d, (v - dt(cam.cy)) / dt(cam.fy) * d, d], 1)
    R, t = scenes.pose_rt(np.asarray(pose, np.float64))
    x = local - t.astype(dt)
    return x @ R.astype(dt), np.abs(local).sum(1) + np.abs(t).sum(), np.log(d / (0.5 * (dt(cam.fx) + dt(cam.fy))))


def _nearest(got, want, slack):
    """got is want rounded to FP32, or the other neighbour where want is within slack of halfway."""
    ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
    return np.abs(got.astype(np.longdouble) - want) <= 0.5 * ulp + slack


# FP64 itself loses about 2^-50 of the terms on the way to a mean, and 2^-52 (|ln| + 1) in a logarithm
@pytest.mark.parametrize("W,H,near,far", [(640, 480, 0.3, 8.0), (1200, 680, 0.3, 8.0), (333, 257, 1e-6, 1e6)])
def test_frames_round_as_from_fp64(W, H, near, far):
    rng = np.random.default_rng(W)
    cam = scenes.Cam(0.82 * W, 0.79 * W, (W - 1) / 2, 0.47 * H, W, H)
    pose = scenes.perturb_pose(scenes.look_at((2.5, 1.5, 0.8), (0.2, 0.1, 1.0)), rng, 20.0, 0.3)
    depth = np.exp(rng.uniform(np.log(near), np.log(far), (H, W))).astype(np.float32)
    depth.flat[::1000] = np.float32(0.805 * W)  # logarithms near zero
    mean, ls = _add(cam, pose, depth)
    m, size, l = _want(cam, pose, depth, np.longdouble)
    assert _nearest(mean, m, 2.0 ** -49 * size[:, None]).all()
    assert _nearest(ls[:, 0], l, 2.0 ** -51 * (np.abs(l) + 1)).all() and (ls == ls[:, :1]).all()


@pytest.mark.parametrize("fx,tx", [(1e-30, 0.0), (3e-38, 0.0), (1e37, 0.0), (1e39, 0.0), (300.0, 1e30), (300.0, 1e39),
                                   (2.0 ** -31, 2.0), (2.0 ** 31, 2.0)])
def test_cameras_outside_the_pairs_range(fx, tx):
    cam = scenes.Cam(fx, fx, 3.5, 3.5, 8, 8)
    depth = np.full((8, 8), 2.0, np.float32)
    mean, ls = _add(cam, [1.0, 0, 0, 0, tx, 0, 0], depth)
    m, _, l = _want(cam, [1.0, 0, 0, 0, tx, 0, 0], depth)
    with np.errstate(over="ignore"):
        np.testing.assert_array_equal(mean, m.astype(np.float32))
    np.testing.assert_array_equal(ls[:, 0], l.astype(np.float32))


def test_columns_beyond_fp32():
    W = (1 << 24) + 11
    cam = scenes.Cam(3e4, 3e4, float(W), 0.0, W, 1)
    depth = np.zeros((1, W), np.float32)
    depth[0, -9:] = 1.0
    mean, _ = _add(cam, [1.0, 0, 0, 0, 0, 0, 0], depth)
    np.testing.assert_array_equal(mean, _want(cam, [1.0, 0, 0, 0, 0, 0, 0], depth)[0].astype(np.float32))
