"""gs_sync_status on another stream than the work's: what is still running on the default stream
is part of the answer, whichever stream the call names."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2408_05635_gb300 import gs, scenes  # noqa: E402


@pytest.mark.parametrize("work,status", [("default", "default"), ("default", "side"), ("side", "side")])
def test_status_follows_the_work(work, status):
    g, cam = scenes.cube_scene(n=2000, seed=1)
    full = gs.GaussianTensors.from_numpy(g)
    half = gs.GaussianTensors(*(getattr(full, k)[:1000].contiguous() for k in ("means", "quats", "log_scales", "logits", "rgb")))
    pose = torch.from_numpy(scenes.identity_pose()).cuda()[None]
    R = gs.Rasterizer()
    prob = R.plan(full, [cam], pose)
    small = R.problem(half.n, [cam], prob.pair_capacity)
    R.render(small, half, pose)
    want = R.sync()
    R.render(prob, full, pose)
    assert R.sync().n_pairs != want.n_pairs
    torch.cuda.synchronize()
    streams = {"default": torch.cuda.default_stream(), "side": torch.cuda.Stream()}
    with torch.cuda.stream(streams[work]):
        torch.cuda._sleep(100_000_000)  # some tens of milliseconds: the pass has not run yet
        R.render(small, half, pose)
    got = R.sync(streams[status])
    assert (got.n_records, got.n_pairs, got.fwd_evals) == (want.n_records, want.n_pairs, want.fwd_evals)
    torch.cuda.synchronize()
    R.close()
