"""An upstream gradient that is not finite at one pixel reaches the Gaussians that contribute to
that pixel and leaves the others' gradients as they are without it."""
import numpy as np
import pytest
import torch

from paper_2408_05635_gb300 import gs, scenes

pytestmark = pytest.mark.gpu
F, W, H = 200.0, 32, 32


def _scene():
    """One 8 x 4 patch: a Gaussian on pixel (1, 1), one on (6, 2) that does not reach it, one between
    pixel centres that the patch lists (its peak is above alpha_min) and no pixel sees."""
    at, z, logit = [(1.0, 1.0), (6.0, 2.0), (3.5, 1.5)], [1.0, 1.2, 1.4], [0.0, 0.0, np.log(0.005 / 0.995)]
    means = [[(u - 15.5) / F * d, (v - 15.5) / F * d, d] for (u, v), d in zip(at, z)]
    g = scenes.Gaussians(np.float32(means), np.tile(np.float32([1, 0.1, 0, 0]), (3, 1)), np.full((3, 3), -9.0, np.float32),
                         np.float32(logit), np.float32([[0.2, 0.3, 0.4]] * 3))
    return gs.GaussianTensors.from_numpy(g), scenes.Cam(F, F, 15.5, 15.5, W, H)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("plane", ["rgb", "depth", "sil"])
@pytest.mark.parametrize("params", [True, False])
def test_only_the_pixels_own_gaussians(plane, value, params):
    gt, cam = _scene()
    pose = torch.from_numpy(scenes.identity_pose()).cuda()[None]
    R = gs.Rasterizer()
    prob = R.plan(gt, [cam], pose)
    res = []
    for v in (0.0, value):
        gen = torch.Generator("cuda").manual_seed(1)
        up = {k: torch.randn(c * W * H, device="cuda", generator=gen) for k, c in (("rgb", 3), ("depth", 1), ("sil", 1))}
        for k in up:
            up[k].reshape(-1, W * H)[:, 1 * W + 1] = 0.0
        up[plane].reshape(-1, W * H)[-1, 1 * W + 1] = v
        R.render(prob, gt, pose)
        res.append(R.backward(gt, upstream=tuple(up.values()), params=params))
        assert R.sync().max_tile == 3
    R.close()
    zero, odd = res
    assert not torch.isfinite(odd["pose_grad"]).all()
    if not params:
        return
    seen = False
    for k, a in odd["grads"].items():
        # the patches' sums meet in atomics, whose order may differ
        torch.testing.assert_close(a[1:], zero["grads"][k][1:], rtol=1e-5, atol=1e-6 * float(zero["grads"][k].abs().max()))
        seen |= not bool(torch.isfinite(a[0]).all())
    assert seen and not bool(zero["grads"]["rgb"][2].any())
