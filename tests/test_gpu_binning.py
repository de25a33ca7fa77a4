"""Tile enumeration of k_project and k_emit on each of its paths -- a block's rows walked by
their own threads or handed out over the block, counted in the block's tile box or in global
memory -- against the oracle (a missed tile loses its pixels' contributions)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from gpu_common import assert_images_close, gpu_render, ocam, params_pair  # noqa: E402
from paper_2408_05635_gb300 import gs, scenes  # noqa: E402


def _scene(kind, n):
    """A cube's Gaussians in random order: a block's records are all over the image."""
    g, _ = scenes.cube_scene(n=n, seed=5)
    ls = g.log_scales.copy()
    if kind == "pixels":  # one or two tiles each
        ls -= ls.mean() + 6.5
    elif kind == "mixed":  # a few span the image (slivers that do: test_row_span.py)
        ls[::97] = 0.0
    return scenes.Gaussians(g.means, g.quats, ls.astype(np.float32), g.logits, g.rgb)


# 8 x 8 tiles: 10,240 of them, more than a block's box holds; 16 x 16: 2,560, inside it; one
# record; a record count one below and one above a block; the last tiles cut
@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("kind", ["pixels", "cube", "mixed"])
@pytest.mark.parametrize("n,size", [(1, (1024, 640)), (255, (1024, 640)), (257, (1021, 635)), (1500, (1024, 640))])
def test_every_tile_is_met(n, size, kind, tile):
    W, H = size
    g = _scene(kind, n)
    cam = scenes.Cam(0.8 * W, 0.8 * W, (W - 1) / 2, (H - 1) / 2, W, H)
    pose = scenes.perturb_pose(scenes.identity_pose(), np.random.default_rng(n), 3.0, 0.05)
    gcfg, op = params_pair()
    R = gs.Rasterizer(gcfg)
    for sub in (1, 4):
        R.set_schedule(tile, tile, sub, 64, 64, 0)
        out, prob, _, counts = gpu_render(R, gs.GaussianTensors.from_numpy(g), [cam], pose[None])
        assert counts.err_flags == 0  # every reserved slot is inside its tile's range
        ref = oracle.render(oracle.Scene(*g.arrays()), ocam(cam), pose, op)
        assert_images_close(out["rgb"].reshape(3, H, W), ref["rgb"], ref["amb"], what="rgb")
        assert_images_close(out["sil"].reshape(H, W), ref["sil"], ref["amb"], what="sil")
    R.close()


def test_capacity_overflow_is_flagged_on_both_paths():
    for tile, kind in [(16, "cube"), (16, "pixels"), (8, "cube"), (8, "pixels")]:
        g = _scene(kind, 1500)
        cam = scenes.Cam(820.0, 820.0, 511.5, 319.5, 1024, 640)
        R = gs.Rasterizer(gs.Config())
        R.set_schedule(tile, tile, 4, 64, 64, 0)
        gt = gs.GaussianTensors.from_numpy(g)
        poses = torch.tensor([scenes.identity_pose()], dtype=torch.float64, device="cuda")
        pairs, _ = R.measure(gt, [cam], poses)
        R.render(R.problem(gt.n, [cam], pairs - 1), gt, poses)
        with pytest.raises(gs.GsError):
            R.sync()
        R.render(R.problem(gt.n, [cam], pairs), gt, poses)
        assert R.sync().n_pairs == pairs
        R.close()
