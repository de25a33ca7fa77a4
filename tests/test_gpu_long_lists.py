"""The per-tile depth order of lists so long that sampled intervals are split again: in one tile
(blocks of 256 threads) and in one of thousands (128), against the device-wide radix sort, bit for
bit, and a second forward on the keys the first one regrouped."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2408_05635_gb300 import gs, scenes  # noqa: E402
from test_gpu_depth_order import _depths, _map, _render  # noqa: E402

CAMS = {"tile": scenes.Cam(60.0, 60.0, 7.5, 7.5, 16, 16), "strip": scenes.Cam(60.0, 60.0, 7.5, 7.5, 65536, 16)}


@pytest.mark.parametrize("cam", sorted(CAMS))
@pytest.mark.parametrize("kind", ["uniform", "wall", "ulps"])
@pytest.mark.parametrize("n", [50_000, 62_000, 100_000, 260_000])
def test_intervals_split_again(n, kind, cam):
    rng = np.random.default_rng(n)
    g = _map(_depths(kind, n, rng), rng, -8.0)
    a, longest = _render(g, CAMS[cam], 0, twice=True)
    b, _ = _render(g, CAMS[cam], gs.GS_SCHED_RADIX)
    assert longest == n
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


def test_capacity_inside_a_long_list():
    """The list is cut at the capacity: flagged, and the context renders right afterwards."""
    n = 100_000
    rng = np.random.default_rng(1)
    gt = gs.GaussianTensors.from_numpy(_map(_depths("uniform", n, rng), rng, -8.0))
    pose = torch.from_numpy(scenes.identity_pose()).cuda()[None]
    R = gs.Rasterizer(gs.Config(alpha_min=1e-6, t_min=0.0))
    full = R.render(R.problem(n, [CAMS["tile"]], n), gt, pose)["rgb"]
    assert R.sync().max_tile == n
    R.render(R.problem(n, [CAMS["tile"]], n - 30_001), gt, pose)
    with pytest.raises(gs.GsError):
        R.sync()
    again = R.render(R.problem(n, [CAMS["tile"]], n), gt, pose)["rgb"]
    assert R.sync().err_flags == 0 and torch.equal(full, again)
    R.close()
