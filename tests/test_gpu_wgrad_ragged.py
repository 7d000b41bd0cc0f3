"""Weight gradient of images whose width is no multiple of 16, or that are at most 8 wide: a value that is not finite
reaches the taps whose pixel lies inside the image and no other weight (integers: every other sum is exact)."""

import numpy as np
import pytest

from oracle import nn

from test_gpu_wgrad_tiles import _bf, _ints

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("chan", [(16, 32), (32, 16), (64, 64), (192, 32)])
@pytest.mark.parametrize("hw", [(1, 1), (6, 6), (1, 8), (8, 8), (17, 5), (9, 9), (12, 12), (5, 17), (8, 24), (7, 40)])
def test_value_that_is_not_finite_stays_in_its_taps(gpu, value, chan, hw):
    torch = pytest.importorskip("torch")
    (h, w), (cin, cout) = hw, chan
    rng = np.random.default_rng(h * 100 + w + cin)
    x, dy = _ints(rng, (2, h, w, cin)), _ints(rng, (2, h, w, cout))
    dy[dy == 0] = 1.0
    for y, x0 in {(0, w - 1), (h - 1, w - 1), (h - 1, 0), (0, 0), (h // 2, w - 1), (h // 2, w // 2)}:
        z = x.copy()
        z[1, y, x0, cin - 3] = 0.0
        ref = nn.conv3x3_wgrad(z, dy)
        z[1, y, x0, cin - 3] = value
        hit = np.zeros(ref.shape, bool)
        for tap in range(9):
            qy, qx = y - (tap // 3 - 1), x0 - (tap % 3 - 1)
            hit[:, tap, cin - 3] = 0 <= qy < h and 0 <= qx < w
        for splits in (1, 3):
            got = gpu.conv3x3_wgrad(_bf(torch, z), _bf(torch, dy), splits=splits).cpu().numpy()
            assert not np.isfinite(got[hit]).any()
            np.testing.assert_array_equal(got[~hit], ref[~hit])
