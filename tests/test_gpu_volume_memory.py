"""Device memory of a loaded volume: words with clearance are held only while a march uses them, voxel_layout 1 and 2
hold one word a voxel, and a volume whose plain words fit is loaded even where its larger words do not."""

import numpy as np
import pytest

from mc_inputs import mono_spectrum
from mc_inputs.tables import MAT_WATER

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _context(gpu, table_path, **opt):
    c = gpu.Context(0, **opt)
    c.load_tables(table_path)
    c.set_spectrum(*mono_spectrum(60.0))
    c.set_geometry(300.0, 600.0, 23, 17, 3.0, 3.0)
    c.load_volume(np.zeros((4, 4, 4), np.uint8), np.ones((4, 4, 4), np.float16), (20.0, 20.0, 20.0))
    c.project([0.3], 1000, 1.0, 1)
    return c


def _volume(torch, n, share):
    """A cube of n^3 voxels of air; in that share of its planes every voxel has a density of its own."""
    mat = torch.zeros((n, n, n), dtype=torch.uint8, device="cuda")
    rho = torch.full((n, n, n), 0.001205, dtype=torch.float16, device="cuda")
    k = int(share * n)
    if k:
        mat[:k] = MAT_WATER
        rho[:k] = (0.8 + 0.4 * torch.rand((k, n, n), device="cuda", generator=torch.Generator("cuda").manual_seed(n))).half()
    return mat, rho


def _free(torch):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


# noise everywhere: neither march uses clearance; noise in a few planes with voxel_layout 1 or 2: none is asked for
@pytest.mark.parametrize("layout,share", [(0, 0.9), (1, 0.05), (2, 0.05), (1, 0.0)])
def test_held_memory(gpu, table_path, layout, share):
    torch = pytest.importorskip("torch")
    n = 192
    mat, rho = _volume(torch, n, share)
    c = _context(gpu, table_path, voxel_layout=layout)
    before = _free(torch)
    c.load_volume(mat, rho, (0.5,) * 3)
    plain = 4 * (n + 8) ** 3
    assert before - _free(torch) <= plain + 8 * MB


def test_clearance_is_given_back(gpu, table_path):
    torch = pytest.importorskip("torch")
    n = 192
    c = _context(gpu, table_path)
    smooth, noisy = _volume(torch, n, 0.05), _volume(torch, n, 0.9)
    before = _free(torch)
    c.load_volume(*smooth, (0.5,) * 3)
    assert before - _free(torch) >= 8 * n**3
    c.load_volume(*noisy, (0.5,) * 3)
    assert before - _free(torch) <= 4 * (n + 8) ** 3 + 16 * MB


# bytes left beside the volume's own arrays, per voxel: room for the staged copy (3) and the plain words (4) with
# little more than that; then for the 64-bit words of a primary-only clearance as well, but not for both
@pytest.mark.parametrize("share,room", [(0.9, 7.5), (0.05, 8.5), (0.35, 13.0)])
def test_volume_that_fits_plainly_is_loaded(gpu, table_path, share, room):
    torch = pytest.importorskip("torch")
    n = 400
    mat, rho = _volume(torch, n, share)
    angles, ref = [0.2, 2.9], None
    for tight in (False, True):
        c = _context(gpu, table_path)
        ballast = None
        if tight:
            ballast = torch.empty(_free(torch) - int(room * n**3) - 64 * MB, dtype=torch.uint8, device="cuda")
        try:
            c.load_volume(mat, rho, (0.25,) * 3)
        finally:
            del ballast
            torch.cuda.empty_cache()
        p = c.project(angles, 1, 0.4, 3, scatter=False)["primary"].cpu().numpy()
        ref = p if ref is None else ref
        np.testing.assert_array_equal(p, ref)
        del c
