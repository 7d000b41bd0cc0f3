"""Up-sampling by rows in shared memory and, where those do not fit, pixel by pixel: the same operations in the same
order, so the same bits.  An image whose left part is another image agrees with it up to where the taps reach past it."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cubic_a", [-0.5, -0.75, -0.6])
@pytest.mark.parametrize("shape", [(64, 256, 256, 2048), (50, 300, 331, 2000), (97, 250, 200, 1250)])
def test_pixel_form_equals_row_form(gpu, cubic_a, shape):
    torch = pytest.importorskip("torch")
    nv, nu, NV, NU = shape
    wide = torch.tensor(np.random.default_rng(NU).normal(size=(3, nv, 4 * nu)), dtype=torch.float32, device="cuda")
    c = gpu.Context(0, denoise_mode=2, cubic_a=cubic_a)
    out = [c.smooth_upsample(im.contiguous(), [0.0, 2.0, 4.0], [1.3, 5.0], W, NV)
           for im, W in ((wide[:, :, :nu], NU), (wide, 4 * NU))]
    # columns whose taps (floor(x) - 1 .. floor(x) + 2) lie inside the narrow image
    keep = int((nu - 3) * NU / nu)
    assert torch.equal(out[0][:, :, :keep], out[1][:, :, :keep])
