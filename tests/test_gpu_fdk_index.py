"""Backprojection of projections too large for 32-bit pixel numbers, or taller than 2^22 rows: the sampled rows are
the right ones (pixel centres at angle 0, as in test_gpu_ramp: the volume is pi times the filtered rows)."""

import numpy as np
import pytest

from oracle import recon

from test_gpu_ramp import SDD, SOD

pytestmark = pytest.mark.gpu

PU = 2.0 ** -5
DU = PU * SOD / SDD


# planes per pixel row (many: eight voxels to a thread) or a few planes far apart (two to a thread)
@pytest.mark.parametrize("nu,nv,nz,step", [(4, 5_000_003, 5_000_003, 1), (4, 5_000_001, 8, 700_000),
                                           (4096, 540_001, 540_001, 1), (4096, 540_001, 8, 76_000)])
def test_rows_far_down_the_panel(gpu, nu, nv, nz, step):
    torch = pytest.importorskip("torch")
    planes = [nz - 2, nz - 3, 1, 0] if step > 1 else [nz - 3, nz - 1000, nz // 2, 7]
    row_of = [int(round((k - 0.5 * (nz - 1)) * step + 0.5 * (nv - 1))) for k in planes]
    if step > 1:
        planes, row_of = planes + [nz - 1], row_of + [int(round(0.5 * (nz - 1) * step + 0.5 * (nv - 1)))]
    assert all(0 <= r < nv - 1 for r in row_of)
    x = np.random.default_rng(nv).uniform(0.5, 1.5, (len(planes), nu)).astype(np.float32)
    p = torch.zeros((1, nv, nu), device="cuda")
    for r, row in zip(row_of, x):
        p[0, r] = torch.from_numpy(row).cuda()
    c = gpu.Context(0)
    c.set_geometry(SOD, SDD, nu, 1, PU, PU * nv)  # the panel of the projections, as one row
    got = c.fdk(p, np.zeros(1, np.float32), nu, nv, (1, nu, nz, 1.0, DU, DU * step))[planes, :, 0].cpu().numpy() / np.pi
    u = (np.arange(nu) - 0.5 * (nu - 1)) * DU
    h = recon.ramlak(nu, DU)
    for k, r in enumerate(row_of):
        v = (r - 0.5 * (nv - 1)) * DU
        w = x[k].astype(np.float64) * SOD / np.sqrt(SOD**2 + u**2 + v * v)
        ref = np.convolve(w, h)[nu - 1:2 * nu - 1] * DU
        assert np.abs(got[k] - ref)[:-1].max() <= 8 * 2.0**-23 * np.abs(w).max() / (4 * DU)
    del p
    torch.cuda.empty_cache()
