"""gs_kernel_times names every kernel of a pass: the depth order is one of its own."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2408_05635_gb300 import gs, scenes  # noqa: E402

BINNING = ["k_project", "k_scan_tiles", "k_emit"]


@pytest.mark.parametrize("flags,order", [(0, "k_sort_tiles"), (gs.GS_SCHED_RADIX, "k_radix_sort")])
def test_the_depth_order_is_named(flags, order):
    g, cam = scenes.cube_scene(n=500, seed=0)
    gt = gs.GaussianTensors.from_numpy(g)
    pose = torch.from_numpy(scenes.identity_pose()).cuda()[None]
    R = gs.Rasterizer()
    R.set_schedule(flags=flags)
    prob = R.plan(gt, [cam], pose)
    gs.gs_set_profiling(R.ctx, True)
    R.render(prob, gt, pose)
    assert [k for k, _ in gs.gs_kernel_times(R.ctx)] == BINNING + [order, "k_forward"]
    gs.gs_set_profiling_mask(R.ctx, ["k_forward", order])
    R.render(prob, gt, pose)
    assert [k for k, _ in gs.gs_kernel_times(R.ctx)] == [order, "k_forward"]
    assert all(ms > 0 for _, ms in gs.gs_kernel_times(R.ctx))
    R.set_schedule(flags=flags | gs.GS_SCHED_FUSED)
    P = cam.width * cam.height
    rgb, depth = torch.rand(3 * P, device="cuda"), torch.rand(P, device="cuda")
    ws, nb = R.workspace(prob)
    adam, loss = torch.zeros(1, 16, dtype=torch.float64, device="cuda"), torch.zeros(1, 1, dtype=torch.float64, device="cuda")
    gs.gs_set_profiling(R.ctx, True)
    gs.gs_track_step(R.ctx, prob, gt.c(), gs.gs_targets(rgb.data_ptr(), depth.data_ptr(), None), pose.clone(), adam, loss, 1, ws, nb)
    assert [k for k, _ in gs.gs_kernel_times(R.ctx)] == BINNING + [order, "k_track_tile", "k_bproject", "k_finalize"]
    R.sync()
    R.close()
