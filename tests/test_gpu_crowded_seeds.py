"""Explicit seeds crowded in a part of a small volume: the layout is chosen for the contours
there are.  Against the bricks and warps of a lattice over the volume (what the planner
tells for its stride), where few CTAs of few warps have hundreds of contours each, it has to
save a fifth of the time at least; the bits are those of the plain path."""
import dataclasses
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim,dims,N,n", [
    (3, (128, 128, 128), 512, 3000),
    (3, (64, 64, 64), 256, 400),
    (2, (512, 512), 128, 20000),
    (2, (180, 180), 64, 3000),
])
def test_crowded_seeds_are_not_taken_for_a_lattice(ndim, dims, N, n):
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(n)
    V = ac.ac_create_volume(rng.integers(0, 200, size=dims[::-1]).astype(np.uint8))
    c = np.zeros((n, 3))
    c[:, :ndim] = rng.random((n, ndim)) * dims * 0.2
    seeds = np.column_stack([c, rng.uniform(2.0, 4.9, n)]).astype(np.float32)
    p = ac.default_params(ndim, 6.0 / math.sqrt(1.5), 170.0, N=N, T=10, seed=3)
    r0 = float(seeds[:, 3].max())
    lattice = ac.ac_plan_layout(ndim, ac.AC_U8, dims, (1.0, 1.0, 1.0), math.sqrt(1.5) * r0, r0, p)
    as_lattice = dataclasses.replace(p, brick=tuple(lattice["brick"]), warps_per_block=lattice["warps_per_block"])
    ms, states = [], []
    for q in (p, as_lattice, dataclasses.replace(p, path=ac.AC_PATH_PLAIN)):
        C = ac.ac_seed(V, explicit=seeds)
        start, best = ac.ac_get_state(C), 1e9
        for _ in range(4):
            ac.ac_set_state(C, start)
            ac.ac_evolve(C, q)
            state = ac.ac_get_state(C)
            best = min(best, ac.ac_evolve_kernel_ms(C))
        ms.append(best)
        states.append(state)
    np.testing.assert_array_equal(states[0], states[2])
    np.testing.assert_array_equal(states[1], states[2])
    assert ms[0] < 0.8 * ms[1]
