"""Where k_project and k_emit choose how a block's tiles are gathered -- in a box of shared
counters or by an atomic a pair, a row by one, four or eight threads -- and where the two choose
differently: every pair counted is written (a capacity of exactly the pairs holds) and every tile
is met (images against the oracle)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from gpu_common import assert_images_close, gpu_render, ocam, params_pair  # noqa: E402
from paper_2408_05635_gb300 import gs, scenes  # noqa: E402


def _scene(kind, n, W, H):
    """Gaussians all over the image, in random order, of a pixel size (or, "wide", 4 rows by
    dozens of columns of tiles; "one": a single large one among pixel-sized ones)."""
    rng = np.random.default_rng(n)
    z = rng.uniform(1.0, 5.0, n)
    xy = rng.uniform(-0.5, 0.5, (n, 2)) * [W, H] / W * z[:, None]
    px = np.full((n, 3), {"pixel": 0.4, "one": 0.4, "ten": 10.0, "forty": 40.0, "wide": 60.0}[kind])
    if kind == "one":
        px[n // 2] = 150.0
    quats = rng.normal(size=(n, 4))
    if kind == "wide":
        px[:, 1:] = 3.0
        quats = np.tile([1.0, 0, 0, 0], (n, 1))
    ls = np.log(px * z[:, None] / W)
    return scenes.Gaussians(np.concatenate([xy, z[:, None]], 1).astype(np.float32), quats.astype(np.float32),
                            ls.astype(np.float32), rng.normal(0, 1, n).astype(np.float32), rng.uniform(size=(n, 3)).astype(np.float32))


# boxes of 1,200 tiles (both kernels'), 3,600 (k_project's only), 5,120 (the same) and 14,400 (neither's)
@pytest.mark.parametrize("W,H,tile", [(640, 480, 16), (1280, 720, 16), (640, 512, 8), (1280, 720, 8)])
@pytest.mark.parametrize("kind,n", [("pixel", 700), ("one", 300), ("ten", 700), ("forty", 257), ("wide", 257)])
def test_every_pair_is_written(kind, n, W, H, tile):
    g = _scene(kind, n, W, H)
    cam = scenes.Cam(float(W), float(W), (W - 1) / 2, (H - 1) / 2, W, H)
    pose = scenes.identity_pose()
    gcfg, op = params_pair()
    gt = gs.GaussianTensors.from_numpy(g)
    poses = torch.from_numpy(pose).cuda()[None]
    ref = oracle.render(oracle.Scene(*g.arrays()), ocam(cam), pose, op)
    R = gs.Rasterizer(gcfg)
    for sub in (1, 4):
        R.set_schedule(tile, tile, sub, 64, 64, 0)
        pairs, _ = R.measure(gt, [cam], poses)
        prob = R.problem(gt.n, [cam], pairs)
        out = R.render(prob, gt, poses)
        assert R.sync().n_pairs == pairs  # and no reservation passed its tile's slots or the capacity
        assert_images_close(out["rgb"].cpu().numpy().reshape(3, H, W), ref["rgb"], ref["amb"], what="rgb")
        assert_images_close(out["sil"].cpu().numpy().reshape(H, W), ref["sil"], ref["amb"], what="sil")
    R.close()
