"""Ramp filter: detector rows of very different size, and rows with pixels far above their others, against FP64 sums.

Two rows share one FP32 transform and a row's pixels share its rounding, so without care a large pixel would show in
its neighbour's row and in its own row's far pixels.  The bounds are those of sums taken row by row and tap by tap:
at the pixel centres (angle 0, power-of-two pitch: the volume is pi times the filtered rows, see test_gpu_ramp) 8 units
of 2^-23 of the row's ordinary largest value over 4 du, and of each large pixel's own contribution."""

import numpy as np
import pytest

from oracle import recon

from test_gpu_ramp import SDD, SOD, _fdk, _rows

pytestmark = pytest.mark.gpu

PU = 2.0 ** -5
DU = PU * SOD / SDD


def _filtered(gpu, p):
    """Filtered rows [nv][nu] of one projection p [1][nv][nu]."""
    _, nv, nu = p.shape
    got = _fdk(gpu, p, np.zeros(1, np.float32), PU, (1, nu, nv, 1.0, DU, DU))
    return got[:, :, 0].astype(np.float64) / np.pi


def _weighted(p):
    _, nv, nu = p.shape
    u = (np.arange(nu) - 0.5 * (nu - 1)) * DU
    v = (np.arange(nv) - 0.5 * (nv - 1)) * DU
    return p[0].astype(np.float64) * SOD / np.sqrt(SOD**2 + u[None] ** 2 + v[:, None] ** 2)


def _check(gpu, p, large):
    """large: the (row, pixel) places of pixels far above their row's others."""
    nu = p.shape[2]
    x, h = _weighted(p), recon.ramlak(nu, DU)
    ref = np.stack([np.convolve(r, h)[nu - 1:2 * nu - 1] * DU for r in x])
    rest = np.abs(x)
    for r, j in large:
        rest[r, j] = 0.0
    bound = np.repeat(rest.max(axis=1, keepdims=True) / (4 * DU), nu, axis=1)
    for r, j in large:
        bound[r] += np.abs(x[r, j] * h[nu - 1 - j:2 * nu - 1 - j]) * DU
    # the last row has no upper neighbour to interpolate with; the last column comes from the mirrored rows
    with np.errstate(over="ignore", invalid="ignore"):
        for got, cols in ((_filtered(gpu, p), slice(None, -1)),
                          (_filtered(gpu, np.ascontiguousarray(p[:, :, ::-1]))[:, ::-1], slice(1, None))):
            assert np.all(np.abs(got - ref)[:-1, cols] <= (8 * 2.0**-23 * bound)[:-1, cols])


@pytest.mark.parametrize("nu", [100, 256, 700, 2048, 4096])
@pytest.mark.parametrize("value", [12.0, 69.0, -1e3, 1e4, 1e6, -1e12, 1e20, 1e29])
def test_large_pixel(gpu, nu, value):
    """One pixel of `value` among line integrals of about 1 (69: a pixel that counts nothing)."""
    for row in (1, 2):
        p = _rows(1, 5, nu, nu)
        p[0, row, nu // 3] = value
        _check(gpu, p, [(row, nu // 3)])


@pytest.mark.parametrize("nu", [129, 1024])
def test_several_large_pixels(gpu, nu):
    p = _rows(1, 7, nu, 3)
    places = [(1, 5), (1, nu // 2), (1, nu - 1), (2, 0), (2, nu // 2), (4, 7)]
    for (r, j), v in zip(places, (1e12, -3e3, 1e6, 5e4, 1e28, -80.0)):
        p[0, r, j] = v
    _check(gpu, p, places)


@pytest.mark.parametrize("nu", [130, 1024])
@pytest.mark.parametrize("scale", [1e-30, 1e-6, 1e-2, 5.0, 1e4, 1e25])
def test_rows_of_different_size(gpu, nu, scale):
    for row in (0, 1, 3):
        p = _rows(1, 5, nu, 11)
        p[0, row] *= np.float32(scale)
        _check(gpu, p, [])


@pytest.mark.parametrize("nu", [2, 90, 1024, 4096])
def test_empty_row_stays_empty(gpu, nu):
    for row in (1, 2):
        p = _rows(1, 5, nu, 2) + np.float32(1.0)
        p[0, row] = 0.0
        _check(gpu, p, [])
        assert not _filtered(gpu, p)[row].any()


@pytest.mark.parametrize("width", [1, 3, 30])
def test_narrow_object(gpu, width):
    """A wire: a few pixels in an empty row, whose even taps are zero."""
    nu = 1024
    p = np.zeros((1, 5, nu), np.float32)
    p[0, 1:4, 500:500 + width] = np.random.default_rng(width).uniform(0.5, 2.0, (3, width))
    _check(gpu, p, [(r, j) for r in (1, 2, 3) for j in range(500, 500 + width)])


# the longest transforms, their last pixel, and the first lengths that are summed directly
@pytest.mark.parametrize("nu", [2, 3, 128, 129, 1024, 2048, 4095, 4096, 4097, 6001])
def test_last_pixel_and_direct_lengths(gpu, nu):
    _check(gpu, _rows(1, 5, nu, nu + 1), [])
