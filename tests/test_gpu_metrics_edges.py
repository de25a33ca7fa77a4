"""gs_image_metrics and gs_msssim where their block and tile edges lie: pixel counts around
a warp, a block and the whole cluster; values outside the range of the FP32 pair sums;
images whose scales leave partial tiles, down to the smallest size."""
import numpy as np
import pytest
import torch

from oracle import metrics as omx
from paper_2408_05635_gb300 import gs

pytestmark = pytest.mark.gpu


def _sums(rgb, depth, rgb_t, depth_t):
    t = [torch.from_numpy(np.ascontiguousarray(a, np.float32).reshape(-1)).cuda() for a in (rgb, depth, rgb_t, depth_t)]
    out = torch.full((4,), -1.0, dtype=torch.float64, device="cuda")
    gs.gs_image_metrics(*t, out)
    again = torch.zeros_like(out)
    gs.gs_image_metrics(*t, again)
    assert torch.equal(out.isnan(), again.isnan()) and torch.equal(out.nan_to_num(), again.nan_to_num())
    return out.cpu().numpy()


def _reference(rgb, depth, rgb_t, depth_t):
    a, b = rgb.astype(np.float32).astype(np.float64), rgb_t.astype(np.float32).astype(np.float64)
    d, t = depth.astype(np.float32).astype(np.float64), depth_t.astype(np.float32).astype(np.float64)
    e = (d - t)[t > 0]
    return np.array([((a - b) ** 2).sum(), np.abs(e).sum(), float(e.size), (e ** 2).sum()])


@pytest.mark.parametrize("pixels", [1, 31, 33, 1023, 1025, 16384, 16385, 16 * 16384 + 5, 40 * 16384 + 7])
def test_image_sums_at_block_edges(pixels):
    rng = np.random.default_rng(pixels)
    rgb, rgb_t = rng.uniform(size=(2, 3, pixels))
    depth, depth_t = rng.uniform(0.5, 4.0, size=(2, pixels))
    depth_t = np.where(rng.uniform(size=pixels) < 0.1, 0.0, depth_t)
    # FP64 sums in another order: a few hundred roundings of 2^-53
    np.testing.assert_allclose(_sums(rgb, depth, rgb_t, depth_t), _reference(rgb, depth, rgb_t, depth_t), rtol=1e-13)


@pytest.mark.parametrize("scale", [1e-20, 1e-13, 1e9, 1e19, 3e30])
def test_image_sums_outside_the_pair_range(scale):
    rng = np.random.default_rng(5)
    rgb, rgb_t = scale * rng.uniform(0.5, 1.0, size=(2, 3, 700))
    depth, depth_t = scale * rng.uniform(0.5, 1.0, size=(2, 700))
    np.testing.assert_allclose(_sums(rgb, depth, rgb_t, depth_t), _reference(rgb, depth, rgb_t, depth_t), rtol=1e-13)


def test_image_sums_of_values_that_are_not_finite():
    rgb, rgb_t = np.full((3, 100), 0.5), np.full((3, 100), 0.25)
    depth, depth_t = np.full(100, 2.0), np.full(100, 1.0)
    rgb[1, 7] = np.inf
    depth[50] = np.nan
    got = _sums(rgb, depth, rgb_t, depth_t)
    assert got[0] == np.inf and np.isnan(got[1]) and got[2] == 100 and np.isnan(got[3])


@pytest.mark.parametrize("W,H", [(176, 176), (177, 207), (200, 181), (511, 187), (193, 700)])
def test_msssim_with_partial_tiles(W, H):
    rng = np.random.default_rng(W)
    a = rng.uniform(size=(3, H, W)).astype(np.float32)
    b = np.clip(a + rng.normal(0, 0.1, a.shape), 0, 1).astype(np.float32)
    out = torch.zeros(4, dtype=torch.float64, device="cuda")
    gs.gs_msssim(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), W, H, out)
    # FP32 window moments: relative rounding of a few 2^-24, averaged over the positions
    np.testing.assert_allclose(out.cpu().numpy()[1:], omx.ms_ssim(b, a)["per_channel"], atol=1e-6)
