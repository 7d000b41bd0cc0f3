"""The transform ramp filter and the tiled backprojection at the sizes where they change form, against the oracle's
direct FP64 sums (the bound of the FDK parity test: 2e-4 of the largest value)."""

import numpy as np
import pytest

from oracle import recon

pytestmark = pytest.mark.gpu

SOD, SDD = 300.0, 600.0


def _rows(n_proj, nv, nu, seed):
    rng = np.random.default_rng(seed)
    u = np.linspace(-1, 1, nu)
    p = 1.5 * np.sqrt(np.clip(1 - (u / 0.7) ** 2, 0, None))[None, None] * rng.uniform(0.5, 1.5, (n_proj, nv, 1))
    return (p + 0.01 * rng.normal(size=p.shape)).astype(np.float32)


def _fdk(gpu, p, angles, pu, grid):
    torch = pytest.importorskip("torch")
    n_proj, nv, nu = p.shape
    c = gpu.Context(0)
    c.set_geometry(SOD, SDD, nu, nv, pu, pu)
    return c.fdk(torch.tensor(p).cuda(), angles, nu, nv, grid).cpu().numpy()


# Row lengths around every transform length (256 .. 8192 points).  At angle 0 the voxels of the plane x = 0 with the
# pitch of the panel at the isocentre sample the pixel centres themselves (a power-of-two pitch: no rounding in their
# positions), so the volume is pi times the filtered rows.  The oracle filters in FP64.  The taps carry up to two
# roundings each and a common one in 1 / pi^2, the weights three, all relative to terms of size max|x| / (4 du); the
# transform works on differences, 100 times smaller: 8 units of 2^-23 of max|x| / (4 du) cover them.
@pytest.mark.parametrize("nu", [2, 3, 127, 128, 129, 256, 257, 512, 513, 1024, 1025, 2048, 2049, 4096])
def test_row_lengths(gpu, nu):
    nv, pu = 5, 2.0 ** -5
    p = _rows(1, nv, nu, nu)
    du = pu * SOD / SDD
    got = _fdk(gpu, p, np.zeros(1, np.float32), pu, (1, nu, nv, 1.0, du, du))[:, :, 0] / np.pi
    u = (np.arange(nu) - 0.5 * (nu - 1)) * du
    v = (np.arange(nv) - 0.5 * (nv - 1)) * du
    x = p[0].astype(np.float64) * SOD / np.sqrt(SOD**2 + u[None] ** 2 + v[:, None] ** 2)
    h = recon.ramlak(nu, du)
    ref = np.stack([np.convolve(r, h)[nu - 1:2 * nu - 1] * du for r in x])
    # the last pixel of a row or column has no right or upper neighbour to interpolate with
    err = np.abs(got - ref)[:-1, :-1]
    assert err.max() <= 8 * 2.0**-23 * np.abs(x).max() / (4 * du)


# one and two voxels per thread column, ragged 16 x 16 tiles, and the deep form (at least 2432 blocks of 8 planes)
@pytest.mark.parametrize("grid", [(1, 1, 1, 1.0, 1.0, 1.0), (17, 33, 3, 2.0, 1.5, 2.0), (130, 259, 131, 0.3, 0.2, 0.4)])
def test_volume_tiles(gpu, grid):
    n_proj, nv, nu = 5, 24, 40
    p = _rows(n_proj, nv, nu, 7)
    angles = (2 * np.pi * np.arange(n_proj) / n_proj).astype(np.float32)
    got = _fdk(gpu, p, angles, 3.0, grid)
    ref = recon.fdk(p.astype(np.float64), angles, 3.0, 3.0, SOD, SDD, grid)
    assert np.abs(got - ref).max() <= 2e-4 * np.abs(ref).max()


def test_chunks_continue(gpu):
    """More projections than one chunk of filtered rows holds (a chunk is 512 MB here: 128 projections)."""
    torch = pytest.importorskip("torch")
    nu, nv, n = 1024, 1024, 130
    p = torch.zeros((n, nv, nu), device="cuda")
    angles = (2 * np.pi * np.arange(n) / n).astype(np.float32)
    sub = _rows(n, 2, nu, 3)
    p[:, 511:513] = torch.tensor(sub).cuda()
    c = gpu.Context(0)
    c.set_geometry(SOD, SDD, nu, nv, 0.2, 0.2)
    got = c.fdk(p, angles, nu, nv, (8, 8, 1, 5.0, 5.0, 1.0)).cpu().numpy()
    ref = recon.fdk(sub.astype(np.float64), angles, 0.2, 0.2, SOD, SDD, (8, 8, 1, 5.0, 5.0, 1.0))
    assert np.abs(got - ref).max() <= 2e-4 * np.abs(ref).max()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 3e38])
def test_bad_row_stays_its_own(gpu, bad):
    """A value that is not finite, or close to overflow, spoils its own detector row only."""
    nu, nv = 130, 8
    p = _rows(1, nv, nu, 5)
    angles = np.array([0.0], np.float32)
    grid = (21, 21, 8, 2.0, 2.0, 0.5 * 0.9)
    clean = _fdk(gpu, p, angles, 0.9, grid)
    for row in (2, 3):
        q = p.copy()
        q[0, row, 40] = bad
        got = _fdk(gpu, q, angles, 0.9, grid)
        # planes whose samples do not touch the row (every plane samples rows within one of its own number) keep their
        # values; the row that shares the transform may round differently (the bound of test_row_lengths, twice)
        for k in range(8):
            if abs(k - row) > 1:
                assert np.abs(got[k] - clean[k]).max() <= 16 * 2.0**-23 * p.max() / (4 * 0.45)
        assert not np.array_equal(got[row], clean[row])
