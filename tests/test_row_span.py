"""row_span (csrc/gs_internal.cuh), the tiles of a tile row that a footprint's support meets, as
an FP32 model in NumPy against every pixel in FP64: round, elongated and sliver footprints
(up to four decades of aspect, tens of thousands of pixels long) inside and beside the image."""
import numpy as np
import pytest

W, H = 1200, 680
f = np.float32


def _span(mx, my, a, b, c, dmax2, ty, tw, th):
    R = f(f(dmax2 * f(1.001)) + f(1e-3))
    w = f(b * b)  # diff_of_products: the products' rounding recovered by fused multiply-adds
    det = f(f(np.float64(a) * np.float64(c) - np.float64(w)) + f(np.float64(w) - np.float64(b) * np.float64(b)))
    aR, ia = f(a * R), f(f(1) / a)
    Y, X = np.sqrt(f(aR / det)), np.sqrt(f(f(R * c) / det))
    t = f(b * np.sqrt(f(R / f(c * det))))
    ly, hy = max(f(f(ty * th) - my), -Y), min(f(f(min((ty + 1) * th - 1, H - 1)) - my), Y)
    if not ly <= hy:
        return 1, 0
    rl, rh = (np.sqrt(max(f(aR - f(det * f(y * y))), f(0))) for y in (ly, hy))
    cl, ch = f(f(-b * ly) * ia), f(f(-b * hy) * ia)
    xr = X if ly <= -t <= hy else max(f(cl + f(rl * ia)), f(ch + f(rh * ia)))
    xl = -X if ly <= t <= hy else min(f(cl - f(rl * ia)), f(ch - f(rh * ia)))
    m = f(f(1e-3) + f(f(4e-7) * max(abs(cl), abs(ch))))
    xl, xr = f(mx + xl), f(mx + xr)
    xl, xr = f(xl - f(m + f(f(1e-6) * abs(xl)))), f(xr + f(m + f(f(1e-6) * abs(xr))))
    lo = max(np.ceil(f(f(xl - f(tw - 1)) * f(1 / tw))), -1)
    hi = min(np.floor(f(xr * f(1 / tw))), 1e7)
    return max(0, int(lo)), min((W - 1) // tw, int(hi))


@pytest.mark.parametrize("tw,th", [(16, 16), (8, 32), (32, 4)])
def test_no_tile_is_missed(tw, th):
    rng = np.random.default_rng(tw)
    u, v = np.arange(W)[None, :], np.arange(H)[:, None]
    met = 0
    for _ in range(250):
        big = 10 ** rng.uniform(0, 4.5)
        small = max(big * 10 ** -rng.uniform(0, 4.2), 0.05)
        th_ = rng.uniform(0, np.pi)
        cs, sn = np.cos(th_), np.sin(th_)
        rot = np.array([[cs, -sn], [sn, cs]])
        S = rot @ np.diag([big ** 2, small ** 2]) @ rot.T
        a, b, c = (f(x / (big * small) ** 2) for x in (S[1, 1], -S[0, 1], S[0, 0]))
        off = rng.normal() * big * 1.5 if rng.random() < 0.6 else 0.0
        mx, my = f(rng.uniform(-50, W + 50) + off * cs), f(rng.uniform(-50, H + 50) + off * sn)
        dmax2 = f(2 * np.log(rng.uniform(0.01, 1.0) * 255))
        if float(a) * float(c) - float(b) ** 2 <= 0:
            continue
        q = float(a) * (u - float(mx)) ** 2 + 2 * float(b) * (u - float(mx)) * (v - float(my)) + float(c) * (v - float(my)) ** 2
        ys, xs = np.nonzero(q <= float(dmax2))
        need = set(zip((ys // th).tolist(), (xs // tw).tolist()))
        spans = {ty: _span(mx, my, a, b, c, dmax2, ty, tw, th) for ty in {y for y, _ in need}}
        met += len(need)
        for y, x in need:
            assert spans[y][0] <= x <= spans[y][1], (big, small, th_, mx, my, y, x, spans[y])
    assert met > 10_000
