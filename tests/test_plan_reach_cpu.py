"""Layouts of small volumes whose regions must be cut (4-byte voxels above all): the planner weighs
that balls of the initial radius leave a region whose halo is shorter than they are, and read
from global memory from the first iteration on, their whole warps with them.  Of these
workloads at most a fifth of the balls may (with the halo's cut weighed by the length of the
run alone it was a third and more)."""
import math

import pytest

from paper_1804_06304_gb300 import ac


@pytest.mark.parametrize("dims,spacing,stride,N", [
    ((178, 152, 39), 1.0, 6.5, 512),
    ((200, 144, 41), 1.0, 6.0, 878),
    ((328, 205, 74), 1.0, 6.0, 512),
    ((363, 253, 93), 1.0, 6.0, 512),
    ((258, 238, 76), 1.0, 6.5, 512),
    ((363, 240, 64), 1.0, 6.5, 512),
    ((179, 143, 51), 1.0, 6.0, 512),
    ((335, 271, 69), 2.0, 6.5, 512),
])
def test_balls_fit_their_regions(dims, spacing, stride, N):
    sp, R0 = (1.0, 1.0, spacing), stride / math.sqrt(1.5)
    p = ac.default_params(3, R0, 100.0, N=N, T=10)
    L = ac.ac_plan_layout(3, ac.AC_F32, dims, sp, stride, R0, p)
    inside = 1.0
    for n, s, b, h in zip(dims, sp, L["brick"], L["halo"]):
        faces = 2.0 - 2.0 / math.ceil(n / b)   # of a brick, within the volume
        out = max(0.0, R0 + 0.5 * p.dR - (h - 1) * s)
        inside *= 1.0 - min(1.0, faces * out / (b * s))
    assert 1.0 - inside <= 0.2, L
