"""gs_image_metrics where its FP32 pairs end: errors whose squares fit FP32 while a thread's
sum of them would not."""
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
