"""Up-sampling with the rows of an output row kept in registers (16-byte stores) against the form that reads them
from shared memory for every row (an output that is not 16-byte aligned takes it): the same operations in the same
order, so the same bits.  Sizes: rows that move on by less than one, by exactly one and by several input rows, a last
block of one row, widths of one and of many 16-byte stores, shared memory just below the 48 KB default."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(33, 20, 300, 1028), (32, 16, 32, 64), (60, 24, 20, 48), (7, 9, 33, 4), (5, 40, 65, 2048),
                                   (64, 40, 64, 300)])
def test_register_rows_equal_shared_rows(gpu, shape):
    torch = pytest.importorskip("torch")
    nv, nu, NV, NU = shape
    imgs = torch.tensor(np.random.default_rng(nv + NU).normal(size=(3, nv, nu)), dtype=torch.float32, device="cuda")
    c = gpu.Context(0, denoise_mode=2)
    outs = []
    for off in (0, 1):
        buf = torch.zeros(2 * NV * NU + 4, dtype=torch.float32, device="cuda")
        out = buf[off:off + 2 * NV * NU].view(2, NV, NU)
        outs.append(c.smooth_upsample(imgs, [0.0, 2.0, 4.0], [1.3, 5.0], NU, NV, out=out).clone())
    assert torch.equal(outs[0], outs[1])
