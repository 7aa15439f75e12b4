"""Bricks of volumes too small for four default bricks per CTA slot: chosen by an
estimate of the launch's time.  The layout must obey the planner's rules, fill its
warps (lanes of a warp that no lattice contour can use are the cost of the old rule),
and leave the results as they are: the plain path, which has no bricks, gives the
same bits."""
import dataclasses
import math

import numpy as np
import pytest

from paper_1804_06304_gb300 import ac

CASES = [   # ndim, dims (x, y, z), voxel type, stride, N
    (3, (64, 64, 32), np.uint8, 4.0, 256),
    (3, (128, 128, 128), np.uint16, 6.0, 512),
    (3, (61, 45, 23), np.float32, 5.0, 100),
    (3, (97, 33, 70), np.float16, 6.5, 48),
    (3, (9, 8, 7), np.uint8, 6.0, 512),
    (2, (512, 512), np.uint8, 6.0, 128),
    (2, (301, 77), np.uint16, 4.0, 100),
    (2, (640, 333), np.float32, 6.0, 300),
    (2, (11, 9), np.float16, 6.0, 40),
]
CODE = {np.uint8: ac.AC_U8, np.uint16: ac.AC_U16, np.float16: ac.AC_F16, np.float32: ac.AC_F32}


def _params(ndim, stride, N, **kw):
    return ac.default_params(ndim, stride / math.sqrt(1.5), 100.0, N=N, T=4, seed=3, **kw)


@pytest.mark.parametrize("ndim,dims,dtype,stride,N", CASES)
def test_layout_of_a_small_volume(ndim, dims, dtype, stride, N):
    R0 = stride / math.sqrt(1.5)
    L = ac.ac_plan_layout(ndim, CODE[dtype], dims, (1.0, 1.0, 1.0), stride, R0, _params(ndim, stride, N))
    G, W = L["lanes_per_contour"], L["warps_per_block"]
    cells = [min(max(1, math.floor(n / stride)), math.ceil(b / stride)) for n, b in zip(dims, L["brick"])]
    full = math.prod(cells)   # contours of a full brick
    assert 1 <= W <= 16
    assert full * G > (W - 1) * 32                       # no warp without a contour in a full brick
    lattice = math.prod(max(1, math.floor(n / stride)) for n in dims)
    if lattice >= 64:
        assert full * G >= 24                            # and at least three quarters of one warp's lanes
    if ndim == 3:
        assert L["smem_bytes"] <= (110 if W <= 8 else 215) * 1024
    else:
        assert L["smem_bytes"] <= 200 * 1024
    assert all(h >= 1 for h in L["halo"][:ndim]) and all(r <= 256 for r in L["region"])


@pytest.mark.gpu
@pytest.mark.parametrize("ndim,dims,dtype,stride,N", CASES)
def test_small_layouts_give_the_plain_paths_bits(ndim, dims, dtype, stride, N):
    vol = np.random.default_rng(N).integers(0, 200, size=dims[::-1]).astype(dtype)
    V = ac.ac_create_volume(vol)
    p = _params(ndim, stride, N)
    out = []
    for path in (ac.AC_PATH_BRICK, ac.AC_PATH_PLAIN):
        C = ac.ac_seed(V, stride=stride)
        ac.ac_evolve(C, dataclasses.replace(p, path=path))
        out.append(ac.ac_get_state(C))
    np.testing.assert_array_equal(out[0], out[1])
