"""Host time of planning a launch: every new handle pays it.  Radii of many voxels, whose halos
do not fit the staged region, cost about what small ones do (a bisection, not a voxel at a
time for every candidate), and the limit on the cut holds as it did step by step."""
import math
import time

import pytest

from paper_1804_06304_gb300 import ac


def _us(dims, stride, N):
    p = ac.default_params(3, stride / math.sqrt(1.5), 100.0, N=N, T=10)
    best = 1e9
    for _ in range(40):
        t = time.perf_counter()
        ac.ac_plan_layout(3, ac.AC_U16, dims, (1.0, 1.0, 1.0), stride, stride / math.sqrt(1.5), p)
        best = min(best, time.perf_counter() - t)
    return 1e6 * best


def test_large_radii_cost_what_small_ones_do():
    assert _us((512, 512, 256), 60.0, 512) < 4.0 * _us((128, 128, 128), 6.0, 512)


@pytest.mark.parametrize("r0,fits", [(1500.0, True), (1700.0, False)])
def test_a_halo_is_cut_by_at_most_4096_voxels(r0, fits):
    """2.5 x 1500 + 3 voxels come down to one within the limit, 2.5 x 1700 + 3 do not."""
    p = ac.default_params(3, r0, 100.0, N=512, T=10, Rmax=4000.0, brick=(8, 8, 8))
    if fits:
        assert ac.ac_plan_layout(3, ac.AC_U8, (900, 900, 900), (1.0, 1.0, 1.0), 6.0, r0, p)["smem_bytes"] <= 110 * 1024
    else:
        with pytest.raises(ac.ACError):
            ac.ac_plan_layout(3, ac.AC_U8, (900, 900, 900), (1.0, 1.0, 1.0), 6.0, r0, p)
