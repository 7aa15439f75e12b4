"""Device voxels repacked into padded rows: rows of any length around the 16-byte chunks
the kernel writes, starting at any element of a larger array, dense and strided, give
what the same voxels give from a dense host array."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ac():
    from paper_1804_06304_gb300 import ac as m
    m.load()
    return m


def _energies(ac, vol, ndim):
    """Energies of balls around every third voxel: they read every voxel of the volume."""
    V = ac.ac_create_volume(vol)
    axes = [np.arange(0, n, 3, dtype=np.float32) for n in vol.shape[::-1]]
    g = np.stack(np.meshgrid(*axes, indexing="ij"), -1).reshape(-1, len(axes))
    seeds = np.concatenate([g, np.zeros((len(g), 3 - ndim), np.float32), np.full((len(g), 1), 2.5, np.float32)], 1)
    C = ac.ac_seed(V, explicit=seeds)
    ac.ac_evolve(C, ac.EvolveParams(N=1, T=1, eps0=0.0, Rmin=0.5, Rmax=9.0, path=ac.AC_PATH_GRID))
    return ac.ac_get_state(C)[4]


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float16, np.float32])
@pytest.mark.parametrize("nx", [2, 3, 7, 15, 17, 31, 33, 50])
@pytest.mark.parametrize("ndim,start", [(2, 0), (2, 1), (3, 0), (3, 1), (3, 3)])
def test_rows_of_any_length_from_any_element(ac, dtype, nx, ndim, start):
    import torch
    rng = np.random.default_rng(nx)
    base = (rng.random((5, 9, nx + 6)) * 200).astype(dtype)
    view = base[1:4, 1:8, start:start + nx] if ndim == 3 else base[2, 1:8, start:start + nx]
    dense = np.ascontiguousarray(view)
    dev = torch.from_numpy(base.view(np.int16) if dtype == np.uint16 else base).cuda()   # 16-bit words as such
    strided = dev[1:4, 1:8, start:start + nx] if ndim == 3 else dev[2, 1:8, start:start + nx]
    flat = torch.empty(dense.size + 5, dtype=dev.dtype, device="cuda")   # dense rows from an odd element
    shifted = flat[start:start + dense.size].view(dense.shape)
    shifted.copy_(strided)
    want = _energies(ac, dense, ndim)
    assert np.any(want != 0)
    np.testing.assert_array_equal(_energies(ac, strided, ndim), want)
    np.testing.assert_array_equal(_energies(ac, shifted, ndim), want)
