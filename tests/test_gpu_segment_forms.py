"""Segmentation and down-sampling in every form their arrays can take (the kernels read aligned arrays in wide words)
and at degenerate histograms, against the oracle: bit for bit, as test_gpu_recon asks at one size."""

import numpy as np
import pytest

from oracle import recon

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("classes", [2, 3])
@pytest.mark.parametrize("shape,off", [((1, 1, 1), 0), ((3, 5, 7), 1), ((16, 16, 16), 2), ((33, 20, 64), 3)])
def test_segment_any_alignment(gpu, table_path, tables, classes, shape, off):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(off + classes)
    lvl = rng.choice(3, size=shape, p=[0.5, 0.35, 0.15])
    vol = (np.array([0.0002, 0.0206, 0.075])[lvl] + rng.normal(0, 0.004, shape)).astype(np.float32)
    buf = torch.zeros(vol.size + 8, device="cuda")
    buf[off:off + vol.size] = torch.from_numpy(vol).cuda().ravel()
    c = gpu.Context(0)
    c.load_tables(table_path)
    mats = (0, 1, 3)[:classes]
    mat, rho, hist, thr = c.segment(buf[off:off + vol.size].view(shape), classes, mats, 0.001205, 60.0, -0.01, 0.09)
    mr = [np.interp(60.0, tables.energies, tables.mu_tot[m]) for m in mats] + [0.0] * (3 - classes)
    m_ref, r_ref, h_ref, t_ref = recon.segment(vol, -0.01, 0.09, classes, mats, mr, 0.001205)
    np.testing.assert_array_equal(hist.astype(np.int64), h_ref)
    np.testing.assert_array_equal(mat.cpu().numpy(), m_ref)
    assert tuple(int(t) for t in thr) == tuple(t_ref)
    got = rho.cpu().numpy().view(np.float16).astype(np.float64)
    assert np.all(np.abs(got - r_ref.astype(np.float16)) <= np.spacing(r_ref.astype(np.float16)).astype(np.float64))


@pytest.mark.parametrize("classes", [2, 3])
@pytest.mark.parametrize("levels", [(0.02,), (0.0, 0.05), (-1.0, 1.0)])
def test_thresholds_of_few_levels(gpu, table_path, classes, levels):
    """Histograms with one or two occupied bins (every threshold pair between them ties: the smallest is taken)."""
    torch = pytest.importorskip("torch")
    vol = np.resize(np.array(levels, np.float32), (5, 6, 8))
    c = gpu.Context(0)
    c.load_tables(table_path)
    _, _, hist, thr = c.segment(torch.from_numpy(vol).cuda(), classes, (0, 1, 3)[:classes], 0.001205, 60.0, -0.01, 0.09)
    h_ref, _ = recon.histogram(vol, -0.01, 0.09)
    np.testing.assert_array_equal(hist.astype(np.int64), h_ref)
    assert tuple(int(t) for t in thr) == tuple(recon.otsu(h_ref, classes))


@pytest.mark.parametrize("off", [0, 1, 2, 4])
def test_bin_volume_any_alignment(gpu, table_path, tables, off):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(off)
    shape = (4, 6, 10)
    n = int(np.prod(shape))
    mat = rng.choice(np.array([0, 1, 3], np.uint8), size=shape)
    rho = (rng.uniform(0.2, 2.5, shape)).astype(np.float16)
    bm = torch.zeros(n + 8, dtype=torch.uint8, device="cuda")
    br = torch.zeros(n + 8, dtype=torch.int16, device="cuda")
    bm[off:off + n] = torch.from_numpy(mat).cuda().ravel()
    br[off:off + n] = torch.from_numpy(rho.view(np.int16)).cuda().ravel()
    c = gpu.Context(0)
    c.load_tables(table_path)
    mo, ro = c.bin_volume(bm[off:off + n].view(shape), br[off:off + n].view(shape), 60.0)
    mr = np.array([np.interp(60.0, tables.energies, tables.mu_tot[m]) for m in range(tables.n_mat)])
    mb, rb = recon.bin_volume(mat, rho.astype(np.float64), mr)
    np.testing.assert_array_equal(mo.cpu().numpy(), mb)
    got = ro.cpu().numpy().view(np.float16).astype(np.float64)
    assert np.all(np.abs(got - rb) <= np.spacing(rb.astype(np.float16)).astype(np.float64))
