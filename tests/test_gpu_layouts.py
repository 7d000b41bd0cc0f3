"""Every layout against bricks over the options of the transport: plain x-fastest words (voxel_layout = 1), and by
default words with clearance of 32 or 64 bits, volumes that both marches or only the primary take by clearance, volumes
that neither does, and volumes beyond L2 (their words stream from HBM and take kernels of their own)."""

import numpy as np
import pytest

from mc_inputs import mono_spectrum
from mc_inputs.tables import MAT_WATER

from test_gpu_clearance import EXACT, _blocks

pytestmark = pytest.mark.gpu

OPTIONS = [dict(), dict(nee_mode=1), dict(doppler=1), dict(nee_mode=1, doppler=1), dict(tally_mode=2), dict(tally_mode=3),
           dict(tally_mode=4, tile_u=8, tile_v=8), dict(tally_mode=2, nee_mode=1, doppler=1), dict(tally_mode=2, doppler=1)]


def _noisy(shape, share):
    rng = np.random.default_rng(int(100 * share))
    mat = np.zeros(shape, np.uint8)
    rho = np.full(shape, 0.001205, np.float16)
    k = int(share * shape[0])
    mat[:k] = MAT_WATER
    rho[:k] = rng.uniform(0.8, 1.2, (k,) + shape[1:]).astype(np.float16)
    return mat, rho


def _images(gpu, table, layout, mat, rho, dv, step, photons, opt):
    c = gpu.Context(0, voxel_layout=layout, **opt)
    c.load_tables(table)
    c.set_spectrum(*mono_spectrum(60.0))
    c.set_geometry(300.0, 600.0, 23, 17, 3.0, 3.0)
    c.load_volume(mat, rho, (dv,) * 3)
    out = c.project([0.0, 0.9, 2.5, 4.1, 5.6], photons, step, 7)
    return out["primary"].cpu().numpy(), out["scatter"].cpu().numpy().astype(np.float64), c.last_stats()


def _agree(gpu, table, layout, mat, rho, dv, step, photons, opt):
    # the walks and the midpoints are the same; the bound of test_gpu_clearance for the sums along a ray
    (pa, sa, ta), (pb, sb, tb) = [_images(gpu, table, l, mat, rho, dv, step, photons, opt) for l in (layout, 2)]
    np.testing.assert_array_equal(pa, pb)
    for k in EXACT:
        assert ta[k] == tb[k], k
    assert np.linalg.norm(sa - sb) <= 2e-5 * np.linalg.norm(sb)


@pytest.mark.parametrize("opt", OPTIONS, ids=str)
@pytest.mark.parametrize("layout,share", [(1, 0.05), (0, 0.05), (0, 0.35), (0, 0.8)])
def test_noise(gpu, variant_table, layout, share, opt):
    mat, rho = _noisy((50, 52, 46), share)
    _agree(gpu, variant_table("bound"), layout, mat, rho, 2.0, 1.1, 20_000, opt)


@pytest.mark.parametrize("opt", OPTIONS, ids=str)
@pytest.mark.parametrize("layout", [0, 1])
def test_blocks(gpu, variant_table, layout, opt):
    mat, rho = _blocks((40, 47, 51))
    _agree(gpu, variant_table("bound"), layout, mat, rho, 1.9, 0.8, 20_000, opt)


# packed words of 97 MB and more: 32-bit words of 300^3, 64-bit words of 232^3 voxels
@pytest.mark.parametrize("opt", [dict(), dict(nee_mode=1), dict(doppler=1)], ids=str)
@pytest.mark.parametrize("layout,n,share", [(0, 300, 0.0), (0, 300, 0.05), (0, 232, 0.05), (1, 300, 0.05)])
def test_beyond_l2(gpu, variant_table, layout, n, share, opt):
    mat, rho = _noisy((n,) * 3, share) if share else _blocks((n,) * 3)
    _agree(gpu, variant_table("bound"), layout, mat, rho, 90.0 / n, 90.0 / n, 20_000, opt)
