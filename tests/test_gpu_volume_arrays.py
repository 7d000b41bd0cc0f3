"""Device arrays that no wide load, or no 2-byte load, may take where they lie: the volume is the same."""

import ctypes as C

import numpy as np
import pytest

from mc_inputs import mono_spectrum

from test_gpu_clearance import _blocks

pytestmark = pytest.mark.gpu


SHAPE = (9, 11, 13)


def _primary(c):
    return c.project([0.4], 1, 1.0, 1, scatter=False)["primary"].cpu().numpy()


@pytest.fixture
def loaded(gpu, table_path):
    mat, rho = _blocks(SHAPE)
    c = gpu.Context(0)
    c.load_tables(table_path)
    c.set_spectrum(*mono_spectrum(60.0))
    c.set_geometry(300.0, 600.0, 23, 17, 3.0, 3.0)
    c.load_volume(mat, rho, (3.0,) * 3)
    return c, mat, rho, _primary(c)


def _load(gpu, c, mat_ptr, rho_ptr):
    nz, ny, nx = SHAPE
    return gpu.library().mc_load_volume(c.h, C.c_void_p(mat_ptr), C.c_void_p(rho_ptr), nx, ny, nz, 3.0, 3.0, 3.0, 1, None)


@pytest.mark.parametrize("off", [0, 1, 3, 5])
def test_densities_at_any_address(gpu, loaded, off):
    torch = pytest.importorskip("torch")
    c, mat, rho, ref = loaded
    m = torch.from_numpy(mat).cuda()
    raw = torch.zeros(2 * mat.size + 16, dtype=torch.uint8, device="cuda")
    raw[off:off + 2 * mat.size] = torch.from_numpy(rho.view(np.uint8).ravel()).cuda()
    torch.cuda.synchronize()
    assert _load(gpu, c, m.data_ptr(), raw.data_ptr() + off) == 0
    np.testing.assert_array_equal(_primary(c), ref)


def test_pinned_arrays(gpu, loaded):
    torch = pytest.importorskip("torch")
    c, mat, rho, ref = loaded
    m, r = torch.from_numpy(mat).pin_memory(), torch.from_numpy(rho).pin_memory()
    assert _load(gpu, c, m.data_ptr(), r.data_ptr()) == 0
    np.testing.assert_array_equal(_primary(c), ref)
