"""Weight gradient at the edges of its tiles: widths around the 8-, 16- and 32-pixel tiles, single rows,
every pairing of channel chunks, more CTAs than tiles.

Inputs are small integers: products and sums (below 2^24) are exact in FP32 whatever their order, so the
result equals the FP64 oracle's.
"""

import numpy as np
import pytest

from oracle import nn

pytestmark = pytest.mark.gpu


def _bf(torch, a):
    return torch.tensor(np.asarray(a, dtype=np.float32)).to(torch.bfloat16).cuda()


def _ints(rng, shape):
    return rng.integers(-4, 5, size=shape).astype(np.float64)


@pytest.mark.parametrize("hw", [(1, 1), (3, 2), (17, 8), (9, 9), (8, 16), (1, 17), (5, 32), (7, 33), (13, 48)])
@pytest.mark.parametrize("chan", [(16, 16), (16, 96), (32, 64), (48, 32), (64, 16), (128, 64), (96, 128)])
def test_exact_at_tile_edges(gpu, hw, chan):
    torch = pytest.importorskip("torch")
    (h, w), (cin, cout) = hw, chan
    rng = np.random.default_rng(h * 1000 + w * 10 + cin + cout)
    x, dy = _ints(rng, (3, h, w, cin)), _ints(rng, (3, h, w, cout))
    ref = nn.conv3x3_wgrad(x, dy)
    for splits in (1, 2, 50):
        got = gpu.conv3x3_wgrad(_bf(torch, x), _bf(torch, dy), splits=splits).cpu().numpy()
        np.testing.assert_array_equal(got, ref, err_msg=str(splits))


@pytest.mark.parametrize("cin", [16, 64])
@pytest.mark.parametrize("at", [(0, 5), (7, 31), (3, 0), (4, 17)])
def test_value_that_is_not_finite_stays_in_its_taps(gpu, cin, at):
    """An infinite input reaches the taps whose pixel lies inside the image and no other weight."""
    torch = pytest.importorskip("torch")
    h, w, cout, (y, x0) = 8, 32, 32, at
    rng = np.random.default_rng(cin + y)
    x, dy = _ints(rng, (1, h, w, cin)), _ints(rng, (1, h, w, cout))
    dy[dy == 0] = 1.0
    x[0, y, x0, 3] = 0.0
    ref = nn.conv3x3_wgrad(x, dy)
    x[0, y, x0, 3] = np.inf
    got = gpu.conv3x3_wgrad(_bf(torch, x), _bf(torch, dy), splits=1).cpu().numpy()
    hit = np.zeros(ref.shape, bool)
    for tap in range(9):
        qy, qx = y - (tap // 3 - 1), x0 - (tap % 3 - 1)
        hit[:, tap, 3] = 0 <= qy < h and 0 <= qx < w
    assert not np.isfinite(got[hit]).any()
    np.testing.assert_array_equal(got[~hit], ref[~hit])
