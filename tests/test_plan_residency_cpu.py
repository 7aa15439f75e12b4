"""The planner counts the CTAs that share an SM's 228 KB by what a CTA really takes: its region,
1 KB that the system reserves and 1 KB of its own variables (rounded up to the region's
alignment).  Workloads whose best layout lies near such a limit get one that keeps to it:
with 64 bytes counted for the variables the planner took regions of up to 960 bytes above,
for a CTA more per SM than there is room for."""
import math

import pytest

from paper_1804_06304_gb300 import ac


@pytest.mark.parametrize("ndim,dims,sz,dtype,stride,N", [
    (2, (2149, 1377, 1), 1.0, ac.AC_U8, 6.5, 64),
    (2, (1173, 1087, 1), 1.0, ac.AC_U16, 6.0, 128),
    (2, (789, 701, 1), 1.0, ac.AC_F32, 5.0, 128),
    (2, (1464, 1125, 1), 1.0, ac.AC_U16, 6.5, 100),
    (3, (128, 80, 28), None, ac.AC_F16, 4.0, 512),
    (3, (68, 49, 25), None, ac.AC_U8, 4.0, 512),
])
def test_layouts_keep_to_the_room_of_an_sm(ndim, dims, sz, dtype, stride, N):
    R0 = stride / math.sqrt(1.5)
    for spacing, T in [(s, T) for s in ([sz] if sz else [1.0, 2.0]) for T in (10, 20)]:
        p = ac.default_params(ndim, R0, 100.0, N=N, T=T)
        L = ac.ac_plan_layout(ndim, dtype, dims, (1.0, 1.0, spacing), stride, R0, p)
        taken = (L["smem_bytes"] + 127) // 128 * 128
        counted = (228 * 1024) // (taken + 1088)   # with 64 bytes for the variables
        by_registers = (16 if ndim == 3 else 21) // L["warps_per_block"]
        assert min(by_registers, counted) <= (228 * 1024) // (taken + 2048)
