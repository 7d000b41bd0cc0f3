"""Down-sampling of voxels whose material is in no table: they add neither mass nor attenuation to their block."""

import numpy as np
import pytest

from oracle import recon

pytestmark = pytest.mark.gpu


def test_unknown_materials_add_nothing(gpu, table_path, tables):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(4)
    shape = (6, 8, 10)
    mat = rng.choice(np.array([0, 1, 3], np.uint8), size=shape)
    rho = rng.uniform(0.2, 2.5, shape).astype(np.float16)
    unknown = rng.random(shape) < 0.3
    unknown[:2, :2, :2] = True  # a block of nothing else
    known = mat.copy()
    mat[unknown] = rng.choice(np.array([tables.n_mat, 7, 8, 9, 31, 32, 128, 255], np.uint8), unknown.sum())
    c = gpu.Context(0)
    c.load_tables(table_path)
    mo, ro = c.bin_volume(torch.from_numpy(mat).cuda(), torch.from_numpy(rho.view(np.int16)).cuda(), 60.0)
    mr = np.array([np.interp(60.0, tables.energies, tables.mu_tot[m]) for m in range(tables.n_mat)])
    mb, rb = recon.bin_volume(known, np.where(unknown, 0.0, rho.astype(np.float64)), mr)
    np.testing.assert_array_equal(mo.cpu().numpy(), mb)
    got = ro.cpu().numpy().view(np.float16).astype(np.float64)
    assert np.all(np.abs(got - rb) <= np.spacing(rb.astype(np.float16)).astype(np.float64))
