"""Long thin footprints through the tile enumeration on the GPU: a tile that the support ellipse
crosses and the row spans miss would leave a hole in it.  tests/test_row_span.py derives the
spans on the CPU; here k_project and k_emit run, a sliver alone (its rows walked by its own thread
or handed out) and several far apart (no tile box)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from gpu_common import gpu_render, ocam, params_pair  # noqa: E402
from paper_2408_05635_gb300 import gs, scenes  # noqa: E402

W, H = 1024, 640


def _slivers(rng, n, aspect):
    """n slivers up to the image's diagonal long, some with their centres outside it, at any angle
    (every third along the rows)."""
    z = rng.uniform(1.0, 4.0, n)
    xy = rng.uniform(-0.7, 0.7, (n, 2)) * [W, H] / W * z[:, None]
    length = np.exp(rng.uniform(np.log(30.0), np.log(400.0), n))
    px = np.stack([length, length / aspect, length / aspect], 1)
    angle = np.where(np.arange(n) % 3 == 0, 0.0, rng.uniform(0, np.pi, n))
    quats = np.stack([np.cos(angle / 2), 0 * angle, 0 * angle, np.sin(angle / 2)], 1)
    ls = np.log(px * z[:, None] / W)
    return scenes.Gaussians(np.concatenate([xy, z[:, None]], 1).astype(np.float32), quats.astype(np.float32),
                            ls.astype(np.float32), np.full(n, 3.0, np.float32), rng.uniform(size=(n, 3)).astype(np.float32))


@pytest.mark.parametrize("tile", [8, 16])
@pytest.mark.parametrize("aspect", [30.0, 1e4])
@pytest.mark.parametrize("n", [1, 6])
def test_no_holes_in_slivers(n, aspect, tile):
    """The oracle's silhouette where it is above 0.3 is found to half of it.  FP32 error of a
    footprint's exponent r away from its centre: the conic's terms are up to r^2 / 0.3 (the dilation
    bounds the thin side), each rounded a few times, 4 * 2^-24 r^2 / 0.3 / 2 = 0.3 at the 900 pixels that
    three deviations of the longest sliver reach inside the image, a factor of 0.74 of an alpha."""
    gcfg, op = params_pair(dilation=0.3)
    cam = scenes.Cam(float(W), float(W), (W - 1) / 2, (H - 1) / 2, W, H)
    pose = scenes.identity_pose()
    R = gs.Rasterizer(gcfg)
    R.set_schedule(tile, tile, 4, 64, 64, 0)
    seen = 0
    for seed in range(6):
        g = _slivers(np.random.default_rng(100 * n + seed), n, aspect)
        out, _, _, counts = gpu_render(R, gs.GaussianTensors.from_numpy(g), [cam], pose[None])
        assert counts.err_flags == 0
        ref = oracle.render(oracle.Scene(*g.arrays()), ocam(cam), pose, op)["sil"]
        sil = out["sil"].reshape(H, W)
        seen += int((ref > 0.3).sum())
        assert (sil[ref > 0.3] > 0.5 * ref[ref > 0.3]).all(), (seed, float((sil - ref).min()))
        assert (ref[sil > 0.3] > 0.5 * sil[sil > 0.3]).all(), (seed, float((sil - ref).max()))
    R.close()
    assert seen > 2000  # the scenes have such pixels (2,113 at least, by the oracle)
