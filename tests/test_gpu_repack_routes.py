"""Voxels that the repack kernel brings into padded rows against voxels that came by row copies
(a host array with gaps between its rows goes up with cudaMemcpy2D, past the kernel): a new
volume and an existing one, from dense host arrays (through a temporary and through the
staging buffer that the volume keeps), from device arrays at any element, dense and with
gaps.  Rows around the 16-byte chunks the kernel writes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _energies(ac, V, shape):
    """Of balls around every third voxel: they read every voxel of the volume."""
    ndim = len(shape)
    g = np.stack(np.meshgrid(*[np.arange(0, n, 3, dtype=np.float32) for n in shape[::-1]], indexing="ij"), -1)
    g = g.reshape(-1, ndim)
    seeds = np.concatenate([g, np.zeros((len(g), 3 - ndim), np.float32), np.full((len(g), 1), 2.5, np.float32)], 1)
    C = ac.ac_seed(V, explicit=seeds)
    ac.ac_evolve(C, ac.EvolveParams(N=1, T=1, eps0=0.0, Rmin=0.5, Rmax=9.0, path=ac.AC_PATH_GRID))
    return ac.ac_get_state(C)[4]


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float16, np.float32])
@pytest.mark.parametrize("nx", [2, 3, 7, 15, 17, 31, 33, 50])
@pytest.mark.parametrize("ndim", [2, 3])
def test_kernel_gives_what_row_copies_give(dtype, nx, ndim):
    import torch
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(nx)
    shape = (7, nx) if ndim == 2 else (3, 7, nx)
    base = (rng.random(shape[:-1] + (nx + 6,)) * 200).astype(dtype)
    gaps = base[..., 1:1 + nx]                 # rows with gaps: copied one by one
    dense = np.ascontiguousarray(gaps)
    want = _energies(ac, ac.ac_create_volume(gaps), shape)
    assert np.ptp(want) > 0
    other = (rng.random(shape) * 200).astype(dtype)
    reloaded = ac.ac_create_volume(other)
    words = base.view(np.int16) if dtype == np.uint16 else base   # 16-bit words as such
    dev = torch.from_numpy(words).cuda()
    flat = torch.empty(dense.size + 5, dtype=dev.dtype, device="cuda")
    for data in [dense, dev[..., 1:1 + nx]] + [flat[s:s + dense.size].view(shape) for s in (0, 1, 3)]:
        if isinstance(data, torch.Tensor) and data.is_contiguous():
            data.copy_(dev[..., 1:1 + nx])
        np.testing.assert_array_equal(_energies(ac, ac.ac_create_volume(data), shape), want)
        ac.ac_load_volume(reloaded, other)
        ac.ac_load_volume(reloaded, data)
        np.testing.assert_array_equal(_energies(ac, reloaded, shape), want)
