"""The reverse walk's sums over a warp's pixels (groups of eight list entries through a
transposed shared matrix, the topmost group partial): list lengths around the group size
and the batch depths, on a tile whose every warp lists every Gaussian, in each tile shape's
warp count, for the full and the pose-only walk, against the oracle; and the fused tracking
kernel against the two-kernel form."""
import numpy as np
import pytest
import torch

import oracle
from gpu_common import assert_grads_close, ocam, params_pair
from paper_2408_05635_gb300 import gs, scenes

pytestmark = pytest.mark.gpu
GRADS = [("means", 0, 3), ("quats", 3, 7), ("log_scales", 7, 10), ("logits", 10, 11), ("rgb", 11, 14)]


def _stack(n):
    """n faint Gaussians over the whole 21 x 19 image, in depth order 1 cm apart (alphas of
    0.02 to 0.04, so 257 of them leave more transmittance than t_min)."""
    rng = np.random.default_rng(n)
    means = np.stack([rng.normal(0, 0.02, n), rng.normal(0, 0.02, n), 1.0 + 0.01 * np.arange(n)], 1)
    opacity = rng.uniform(0.02, 0.04, n)
    g = scenes.Gaussians(means.astype(np.float32), rng.normal(size=(n, 4)).astype(np.float32),
                         rng.normal(-0.5, 0.2, (n, 3)).astype(np.float32),
                         np.log(opacity / (1 - opacity)).astype(np.float32),
                         rng.uniform(size=(n, 3)).astype(np.float32))
    return g, scenes.Cam(30.0, 31.0, 10.0, 9.0, 21, 19)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 63, 64, 65, 255, 256, 257])
@pytest.mark.parametrize("sched", [(16, 16, 4, 256, 256), (8, 8, 1, 64, 64), (32, 8, 2, 256, 128)])
def test_gradients_of_a_stack(n, sched):
    g, cam = _stack(n)
    gcfg, op = params_pair()
    pose = scenes.identity_pose()
    sc, oc = oracle.Scene(*g.arrays()), ocam(cam)
    amb = oracle.render(sc, oc, pose, op)["amb"]
    rng = np.random.default_rng(1000 + n)
    H, W = cam.height, cam.width
    up = [np.where(amb[None], 0.0, rng.normal(size=(3, H, W))), np.where(amb, 0.0, rng.normal(size=(H, W))),
          np.where(amb, 0.0, rng.normal(size=(H, W)))]
    ref = oracle.backward(sc, oc, pose, op, *up)
    ups = tuple(torch.tensor(a.reshape(-1).astype(np.float32), device="cuda") for a in up)
    gt = gs.GaussianTensors.from_numpy(g)
    poses = torch.tensor(pose[None], dtype=torch.float64, device="cuda")
    R = gs.Rasterizer(gcfg)
    R.set_schedule(*sched)
    prob = R.plan(gt, [cam], poses)
    R.render(prob, gt, poses)
    full = R.backward(gt, upstream=ups)
    counts = R.sync()
    assert counts.err_flags == 0 and counts.max_tile == n and counts.bwd_contrib > 0
    R.render(prob, gt, poses)
    only = R.backward(gt, upstream=ups, params=False)
    R.close()
    for name, lo, hi in GRADS:
        assert_grads_close(full["grads"][name].cpu().numpy().reshape(n, -1), ref["grads"][:, lo:hi], what=name)
    assert_grads_close(full["pose_grad"].cpu().numpy()[0], ref["pose6"], what="pose")
    assert_grads_close(only["pose_grad"].cpu().numpy()[0], ref["pose6"], what="pose only")


@pytest.mark.parametrize("n", [1, 8, 9, 256, 257, 520])
def test_fused_kernel_on_a_stack(n):
    """520: three batches, the forward ending in the last one (alphas of a stack this deep
    stop some pixels early, so the warps enter the reverse walk from different batches)."""
    g, cam = _stack(n)
    gcfg, _ = params_pair(sil_thresh=0.0)
    P = cam.width * cam.height
    rng = np.random.default_rng(n)
    tgt = [torch.tensor(a.astype(np.float32), device="cuda") for a in
           (rng.uniform(size=3 * P), rng.uniform(0.5, 2.0, size=P), rng.uniform(0.5, 2.0, size=P))]
    gt = gs.GaussianTensors.from_numpy(g)
    start = torch.tensor(scenes.identity_pose()[None], dtype=torch.float64, device="cuda")
    res = []
    for flags in (0, gs.GS_SCHED_FUSED):
        R = gs.Rasterizer(gcfg)
        R.set_schedule(flags=flags)
        prob = R.plan(gt, [cam], start)
        ws, nb = R.workspace(prob)
        pose, adam = start.clone(), torch.zeros(1, 16, dtype=torch.float64, device="cuda")
        hist = torch.zeros(1, 1, dtype=torch.float64, device="cuda")
        gs.gs_track_step(R.ctx, prob, gt.c(), gs.gs_targets(*(t.data_ptr() for t in tgt)), pose, adam, hist, 1, ws, nb)
        c = R.sync()
        st = adam.cpu().numpy()[0]
        res.append((hist.item(), np.concatenate([st[0:3], st[6:9]]) / 0.1,
                    (c.fwd_evals, c.fwd_contrib, c.bwd_evals, c.bwd_contrib)))
        R.close()
    (l0, g0, c0), (l1, g1, c1) = res
    assert l1 == l0 and c1 == c0 and c0[3] > 0  # the forward is the same arithmetic
    assert np.abs(g1 - g0).max() <= 1e-5 * np.abs(g0).max(), (g0, g1)
