"""gs_map_add and gs_map_prune at the edges of their 1,024-item blocks: item counts around a
block, blocks that keep all, none or some of their items, every storage form, a capacity that
ends inside a block; and the unprojection at depths inside and outside the range of its FP32
pairs.  Moved values bit for bit; unprojected means and log-scales within one unit in the
last place of the FP64 values rounded to FP32 (the pairs carry about 2^-30 or better)."""
import numpy as np
import pytest
import torch

from paper_2408_05635_gb300 import gs, scenes

pytestmark = pytest.mark.gpu
FORMS = [(None, False), (torch.bfloat16, False), (torch.float16, True)]


def _random_map(cap, n, lowp, iso, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    m = gs.Map(cap, lowp_dtype=lowp, isotropic=iso)
    for k in m.GROUPS:
        m.p[k].copy_(torch.randn(m.p[k].shape, device="cuda", generator=gen))
        if lowp is not None and k != "means":
            m.lp[k].copy_(torch.randn(m.p[k].shape, device="cuda", generator=gen))
    m.state.copy_(torch.randn(m.state.shape, device="cuda", generator=gen))
    m.count.fill_(n)
    return m


def _moments(m):
    out, off, per = {}, 0, sum(m.WIDTH[k] for k in m.GROUPS)
    for k in m.GROUPS:
        w, c = m.WIDTH[k], m.capacity
        out[k] = [m.state[(b + off) * c:(b + off + w) * c].reshape(c, w) for b in (0, per)]
        off += w
    return out


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 3000])
@pytest.mark.parametrize("keep", ["all", "none", "some"])
@pytest.mark.parametrize("lowp,iso", FORMS)
def test_prune_moves_every_value(n, keep, lowp, iso):
    src, dst = _random_map(3000, n, lowp, iso, 1), _random_map(3004, 7, lowp, iso, 2)
    kept = {"all": torch.ones, "none": torch.zeros}.get(keep, lambda s, device: torch.rand(s, device=device) < 0.6)(n, device="cuda").bool()
    src.p["logits"][:n] = torch.where(kept, 1.0, -9.0)
    before = {k: v.clone() for k, v in dst.p.items()}
    src.prune_into(dst)
    c = int(kept.sum())
    assert dst.n == c
    at = kept.nonzero()[:, 0]
    for k in src.GROUPS:
        assert torch.equal(dst.p[k][:c], src.p[k][at]) and torch.equal(dst.p[k][c:], before[k][c:])
        if lowp is not None and k != "means":
            assert torch.equal(dst.lp[k][:c], src.lp[k][at])
        for a, b in zip(_moments(src)[k], _moments(dst)[k]):
            assert torch.equal(b[:c], a[at])


@pytest.mark.parametrize("W,H", [(31, 33), (32, 32), (41, 25), (53, 59)])
@pytest.mark.parametrize("lowp,iso", FORMS)
@pytest.mark.parametrize("short", [0, 300])
def test_add_writes_every_value(W, H, lowp, iso, short):
    rng = np.random.default_rng(W)
    cam = scenes.Cam(0.7 * W, 0.75 * W, 0.45 * W, 0.55 * H, W, H)
    pose = scenes.perturb_pose(scenes.look_at((2.5, 1.5, 0.8), (0.2, 0.1, 1.0)), rng, 20.0, 0.3)
    depth = np.exp(rng.uniform(np.log(1e-3), np.log(1e3), (H, W))).astype(np.float32)
    depth[rng.uniform(size=(H, W)) < 0.2] = 0.0
    depth.flat[:4] = [1e-25, 1e25, 1e-38, 3e38]
    rgb = rng.uniform(size=(3, H, W)).astype(np.float32)
    n0, P = 5, int((depth > 0).sum())
    cap = (n0 + P + 3) // 4 * 4 - (short + 3) // 4 * 4
    m = _random_map(cap, n0, lowp, iso, 3)
    old = {k: v[:n0].clone() for k, v in m.p.items()}
    m.add_from_frame(cam, torch.tensor(pose, device="cuda"), torch.tensor(rgb, device="cuda"), torch.tensor(depth, device="cuda"))
    n1 = min(n0 + P, cap)
    assert m.n == n1 and m.err.item() == (1 if n0 + P > cap else 0)
    v, u = [a[:n1 - n0].astype(np.float64) for a in np.nonzero(depth > 0)]
    d = depth[depth > 0][:n1 - n0].astype(np.float64)
    local = np.stack([(u - cam.cx) / cam.fx * d, (v - cam.cy) / cam.fy * d, d], 1)
    R, t = scenes.pose_rt(pose)
    with np.errstate(over="ignore"):
        want = {"means": (local - t) @ R, "log_scales": np.log(d / (0.5 * (cam.fx + cam.fy)))[:, None].repeat(m.WIDTH["log_scales"], 1),
                "logits": np.zeros(len(d)), "rgb": rgb.reshape(3, -1)[:, depth.reshape(-1) > 0].T[:len(d)],
                "quats": np.tile([1.0, 0, 0, 0], (len(d), 1))}
        for k in m.GROUPS:
            assert torch.equal(m.p[k][:n0], old[k])
            got, ref = m.p[k][n0:n1].cpu().numpy().astype(np.float64), want[k].astype(np.float32)
            ulp = np.spacing(np.abs(ref)).astype(np.float64)
            if k == "means":  # R^T (x_c - t) cancels: pairs carry 2^-43 of the terms
                ulp += 2.0 ** -43 * (np.abs(local - t).sum(1, keepdims=True) + np.abs(t).sum())
            ref = ref.astype(np.float64)
            same = np.isinf(ref) & (got == ref)
            assert (same | (np.abs(got - ref) <= ulp)).all(), (k, np.abs(got - ref).max())
            if lowp is not None and k != "means":
                assert torch.equal(m.lp[k][n0:n1], m.p[k][n0:n1].to(lowp))
    for k in m.GROUPS:
        assert all((x[n0:n1] == 0).all() for x in _moments(m)[k])
