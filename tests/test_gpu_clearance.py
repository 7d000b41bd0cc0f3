"""Volumes with clearance (many midpoints from one word) against the same volume marched step by step.

The default layout takes every midpoint inside a uniform cube from one word where the volume allows it; bricks
(voxel_layout = 2) always gather each midpoint.  The midpoints are the same, so the primary's integer column masses,
the walks and every step count agree exactly, and the scatter image differs only by the order of FP32 sums of one
optical depth: a few hundred terms of one sign, each rounded to 2^-24, and exp of the result (|tau| up to ~20).
"""

import numpy as np
import pytest

from mc_inputs import mono_spectrum
from mc_inputs.tables import MAT_AL, MAT_WATER

pytestmark = pytest.mark.gpu

EXACT = ("histories", "flight_steps", "nee_steps", "nee_rays", "photo", "compton", "rayleigh", "escape")


def _pair(gpu, table_path, mat, rho, dv, panel=(23, 17, 3.0), **opt):
    out = []
    for layout in (0, 2):
        c = gpu.Context(0, voxel_layout=layout, **opt)
        c.load_tables(table_path)
        c.set_spectrum(*mono_spectrum(60.0))
        c.set_geometry(300.0, 600.0, panel[0], panel[1], panel[2], panel[2])
        c.load_volume(mat, rho, dv)
        out.append(c)
    return out


def _same(gpu, ctxs, step, photons=20_000):
    angles = [0.0, 0.9, 2.5, 4.1, 5.6]  # every octant of directions
    (a, b), st = [c.project(angles, photons, step, 7) for c in ctxs], [c.last_stats() for c in ctxs]
    np.testing.assert_array_equal(a["primary"].cpu().numpy(), b["primary"].cpu().numpy())
    for k in EXACT:
        assert st[0][k] == st[1][k], k
    x, y = (t["scatter"].cpu().numpy().astype(np.float64) for t in (a, b))
    assert np.linalg.norm(x - y) <= 2e-5 * np.linalg.norm(y)
    return st[0]


def _blocks(shape, dens=(0.001205, 1.0, 2.7), seed=3):
    """Large uniform blocks of three materials."""
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    mat = np.zeros(shape, np.uint8)
    for m in (MAT_WATER, MAT_AL, MAT_WATER):
        lo = [int(rng.integers(0, max(1, n // 2))) for n in shape]
        hi = [min(n, l + max(1, n // 3)) for l, n in zip(lo, shape)]
        mat[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] = m
    rho = np.choose(np.minimum(mat, 2), dens).astype(np.float16)
    return mat, rho


@pytest.mark.parametrize("shape,dv,step", [((1, 1, 1), (40.0, 40.0, 40.0), 3.0), ((2, 1, 3), (20.0, 30.0, 11.0), 40.0),
                                           ((31, 33, 62), (2.0, 2.5, 1.5), 0.7), ((64, 30, 130), (1.0, 2.0, 0.7), 0.31),
                                           ((140, 136, 133), (0.6, 0.6, 0.6), 0.6)])
def test_clearance_matches_steps(gpu, table_path, shape, dv, step):
    mat, rho = _blocks(shape)
    _same(gpu, _pair(gpu, table_path, mat, rho, dv), step)


@pytest.mark.parametrize("opt", [dict(nee_mode=1), dict(tally_mode=4, tile_u=8, tile_v=8), dict(tally_mode=3),
                                 dict(n_split=1, rr_threshold=1e-9), dict(use_graph=1)])
def test_clearance_options(gpu, table_path, opt):
    mat, rho = _blocks((40, 47, 51))
    ctxs = _pair(gpu, table_path, mat, rho, (1.7, 1.9, 2.1), **opt)
    st = _same(gpu, ctxs, 0.8)
    assert st["nee_rays"] > 0


@pytest.mark.parametrize("opt", [dict(), dict(nee_mode=1), dict(tally_mode=4, tile_u=8, tile_v=8)])
@pytest.mark.parametrize("share", [0.05, 0.35])
def test_many_pairs(gpu, table_path, share, opt):
    """More pairs than a palette names (a core with a density of its own in every voxel): 64-bit words.  At the larger
    share the primary alone marches by clearance."""
    rng = np.random.default_rng(2)
    shape = (50, 52, 46)
    mat = np.zeros(shape, np.uint8)
    rho = np.full(shape, 0.001205, np.float16)
    y, x = np.meshgrid(np.linspace(-1, 1, 52), np.linspace(-1, 1, 46), indexing="ij")
    core = np.broadcast_to(x * x + y * y < 4 * share / np.pi, shape)
    mat[core] = MAT_WATER
    rho[core] = rng.uniform(0.8, 1.2, core.sum()).astype(np.float16)
    _same(gpu, _pair(gpu, table_path, mat, rho, (2.0, 1.8, 2.2), **opt), 1.1)


@pytest.mark.parametrize("pairs", [255, 256, 257])
def test_palette_edges(gpu, table_path, pairs):
    """The distinct (material, density) pairs around the 256 a word's palette index can name: a thin layer holds
    them, the rest is uniform."""
    mat, rho = _blocks((48, 44, 60), dens=(0.001205, 1.0, 2.7))
    extra = pairs - len(np.unique(np.stack([mat.ravel().astype(np.int64), rho.view(np.uint16).ravel()], 1), axis=0))
    line = np.float16(0.5) + np.arange(extra) * np.float16(2.0) ** -11
    flat = np.arange(extra)
    mat[0].ravel()[flat] = MAT_WATER
    rho[0].ravel()[flat] = line.astype(np.float16)
    assert len(np.unique(np.stack([mat.ravel().astype(np.int64), rho.view(np.uint16).ravel()], 1), axis=0)) == pairs
    _same(gpu, _pair(gpu, table_path, mat, rho, (2.0, 2.0, 2.0)), 1.0)


def test_volume_arrays_anywhere(gpu, table_path):
    """Device arrays at any address (the load reads aligned ones in wide words) and host arrays give the same volume;
    bad voxels anywhere in them are found."""
    torch = pytest.importorskip("torch")
    shape = (9, 11, 13)
    mat, rho = _blocks(shape)
    n = mat.size
    ref = None
    for off in (None, 0, 1, 3):
        if off is None:
            m, r = mat, rho
        else:
            bm = torch.zeros(n + 8, dtype=torch.uint8, device="cuda")
            br = torch.zeros(n + 8, dtype=torch.float16, device="cuda")
            bm[off:off + n] = torch.from_numpy(mat).cuda().ravel()
            br[off:off + n] = torch.from_numpy(rho).cuda().ravel()
            m, r = bm[off:off + n].view(shape), br[off:off + n].view(shape)
        c = _pair(gpu, table_path, m, r, (3.0, 3.0, 3.0))[0]
        p = c.project([0.4], 1, 1.0, 1, scatter=False)["primary"].cpu().numpy()
        ref = p if ref is None else ref
        np.testing.assert_array_equal(p, ref)
        if off is not None:
            for at in (0, 7, n - 1):
                keep = m.view(-1)[at].clone()
                m.view(-1)[at] = 200
                with pytest.raises(gpu.MCError, match="INVALID_ARG"):
                    c.load_volume(m, r, (3.0, 3.0, 3.0))
                m.view(-1)[at] = keep
                keep = r.view(-1)[at].clone()
                for bad in (-1.0, float("inf"), float("nan")):
                    r.view(-1)[at] = bad
                    with pytest.raises(gpu.MCError, match="INVALID_ARG"):
                        c.load_volume(m, r, (3.0, 3.0, 3.0))
                r.view(-1)[at] = keep
