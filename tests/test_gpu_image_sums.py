"""gs_image_metrics' sums on the FP32 pipes: errors whose squares fit FP32 while a thread's sum
of them would not, and a frame's sums against exact ones."""
import math

import numpy as np
import pytest
import torch

from paper_2408_05635_gb300 import gs

pytestmark = pytest.mark.gpu


# 21 pixels a thread, a frame, a very large image; 2^40 is where the pairs' range ends
@pytest.mark.parametrize("error", [np.nextafter(np.float32(2.0 ** 40), np.float32(0)), 2.0 ** 40, 1e15, 3e17, 9e17, 2.0 ** 59])
@pytest.mark.parametrize("pixels", [20 * 16384 + 5, 640 * 480, 4096 * 4096])
def test_image_sums_of_large_errors(pixels, error):
    e = float(np.float32(error))
    rgb, depth = (torch.full((k * pixels,), e, device="cuda") for k in (3, 1))
    zero, tiny = torch.zeros(3 * pixels, device="cuda"), torch.full((pixels,), 1e-30, device="cuda")
    out = torch.zeros(4, dtype=torch.float64, device="cuda")
    gs.gs_image_metrics(rgb, depth, zero, tiny, out)
    # FP64 sums of equal terms: up to 3 x 1024 roundings in a thread, a few tens across
    np.testing.assert_allclose(out.cpu().numpy(), [3 * pixels * e * e, pixels * e, pixels, pixels * e * e], rtol=1e-12)


def _square(e):
    """e^2 as two FP64 values that add to it exactly (Veltkamp's split, Dekker's product)."""
    c = e * 134217729.0
    h = c - (c - e)
    l = e - h
    p = e * e
    return np.concatenate([p, ((h * h - p) + 2 * h * l) + l * l])


@pytest.mark.parametrize("noise", [None, 0.01, 1e-4])
@pytest.mark.parametrize("W,H", [(333, 257), (640, 480), (1200, 680)])
def test_frame_sums_within_a_few_roundings(W, H, noise):
    """Against exactly rounded sums (the differences of FP32 values near 1 are exact in FP64).
    Bound: 4 + 5 + 16 FP64 additions at most between eight threads' sums and the result, each
    half a unit of 2^-52, and 1 more for the squares' low parts (2^-49 of each, either sign, over
    hundreds of thousands of squares)."""
    for seed in range(3):
        rng = np.random.default_rng(seed)
        a = rng.uniform(size=3 * W * H).astype(np.float32)
        b = (rng.uniform(size=a.size) if noise is None else a + noise * rng.normal(size=a.size)).astype(np.float32)
        d = rng.uniform(0.5, 5.0, W * H).astype(np.float32)
        t = (d * (1 + 0.005 * rng.normal(size=d.size))).astype(np.float32)
        t[rng.uniform(size=t.size) < 0.05] = 0
        out = torch.zeros(4, dtype=torch.float64, device="cuda")
        gs.gs_image_metrics(*(torch.from_numpy(x).cuda() for x in (a, d, b, t)), out)
        ec = a.astype(np.float64) - b.astype(np.float64)
        ed = (d.astype(np.float64) - t.astype(np.float64))[t > 0]
        want = [math.fsum(_square(ec)), math.fsum(np.abs(ed)), float(ed.size), math.fsum(_square(ed))]
        np.testing.assert_allclose(out.cpu().numpy(), want, rtol=26 * 2.0 ** -53)
