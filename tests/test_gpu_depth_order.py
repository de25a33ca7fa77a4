"""The per-tile depth order (k_sort_tiles) over list lengths at the edges of its paths and
over depth distributions that spread, crowd or tie, against the device-wide radix sort
(bit-identical images) and, where every depth ties, against the closed form of Eq. 2."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2408_05635_gb300 import gs, scenes  # noqa: E402


def _depths(kind, n, rng):
    if kind == "uniform":
        return rng.uniform(0.5, 9.0, n)
    if kind == "wall":  # most of the list within a few mm, some far behind
        return np.where(rng.random(n) < 0.8, 3.0 + 0.002 * rng.normal(size=n), rng.uniform(0.4, 300.0, n))
    if kind == "geometric":
        return np.exp(rng.uniform(np.log(0.3), np.log(1e4), n))
    return 2.0 + rng.integers(0, max(n // 3, 1), n) * 2.0 ** -22  # "ulps": neighbours and pairs that tie


def _map(z, rng, logit):
    """Gaussians on the optical axis whose footprint is 18 px wide at any depth."""
    n = z.size
    means = np.zeros((n, 3), np.float32)
    means[:, 2] = z
    ls = np.repeat(np.log(0.3 * z)[:, None], 3, 1).astype(np.float32)
    return scenes.Gaussians(means, np.tile(np.float32([1, 0, 0, 0]), (n, 1)), ls, np.full(n, logit, np.float32),
                            rng.uniform(size=(n, 3)).astype(np.float32))


def _render(g, cam, flags, twice=False):
    # no early stop, so every entry of every list counts
    R = gs.Rasterizer(gs.Config(alpha_min=1e-6, t_min=0.0))
    R.set_schedule(flags=flags)
    gt = gs.GaussianTensors.from_numpy(g)
    pose = torch.tensor([scenes.identity_pose()], dtype=torch.float64, device="cuda")
    prob = R.plan(gt, [cam], pose, margin=1.1)
    out = R.render(prob, gt, pose)
    if twice:  # the order is made again from the same keys
        again = {k: torch.empty_like(v) for k, v in out.items()}
        gs.gs_forward(R.ctx, None, again["rgb"], again["depth"], again["sil"], None)
        for k in out:
            assert torch.equal(out[k], again[k]), k
    counts = R.sync()
    assert counts.err_flags == 0
    R.close()
    return {k: v.cpu().numpy() for k, v in out.items()}, int(counts.max_tile)


# one tile: long lists per tile; 128 tiles of which a few are full: the other block size
CAMS = {"tile": scenes.Cam(60.0, 60.0, 7.5, 7.5, 16, 16), "strip": scenes.Cam(60.0, 60.0, 7.5, 7.5, 2048, 16)}


@pytest.mark.parametrize("cam", sorted(CAMS))
@pytest.mark.parametrize("kind", ["uniform", "wall", "geometric", "ulps"])
@pytest.mark.parametrize("n", [1, 2, 33, 127, 129, 1023, 1024, 1025, 2300, 9000])
def test_lists_in_radix_order(n, kind, cam):
    rng = np.random.default_rng(n)
    g = _map(_depths(kind, n, rng), rng, -8.0)
    a, longest = _render(g, CAMS[cam], 0, twice=True)
    b, _ = _render(g, CAMS[cam], gs.GS_SCHED_RADIX)
    assert longest == n
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


def test_more_keys_than_the_sample_sort_takes():
    rng = np.random.default_rng(3)
    g = _map(_depths("uniform", 66_000, rng), rng, -8.0)
    a, longest = _render(g, CAMS["tile"], 0, twice=True)
    b, _ = _render(g, CAMS["tile"], gs.GS_SCHED_RADIX)
    assert longest == 66_000
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("cam", sorted(CAMS))
@pytest.mark.parametrize("n", [200, 1024, 1500, 5000])
def test_tied_depths_in_index_order(n, cam):
    """All depths equal: at the pixel beside the common centre every footprint has the same
    alpha a, and Eq. 2 is sum_i c_i a (1 - a)^i in index order.  FP32 error: (1 - a)^i carries
    i (u + da) with u = 2^-24 and da the footprint's, below 1e-6 here; weighted by a (1 - a)^i
    that sums to at most (u + da) / a = 1.1e-4, and a wrong order differs by about
    sd(c) sqrt(a / 2) = 0.02."""
    rng = np.random.default_rng(n)
    g = _map(np.full(n, 2.0), rng, np.log(0.01 / 0.99))
    out, longest = _render(g, CAMS[cam], 0)
    assert longest == n
    c = CAMS[cam]
    px = out["rgb"].reshape(3, c.height, c.width)[:, 7, 7]
    # the centre (7.5, 7.5) is half a pixel away in x and y; the footprint is 60 * 0.3 px wide
    a = 0.01 * np.exp(-0.5 * (0.25 + 0.25) / 18.0 ** 2)
    w = a * (1 - a) ** np.arange(n)
    np.testing.assert_allclose(px, (w[:, None] * g.rgb.astype(np.float64)).sum(0), atol=1.5e-4, rtol=0)
