"""The layout of a launch over several volumes follows from all of them, whatever their order:
with a small volume first, in the middle or last the same balls stay in the staged regions
(the path counters), and every set evolves to the same bits."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim,dims,spacings,N", [
    (3, [(24, 20, 12), (96, 96, 48), (96, 96, 48), (70, 90, 33)], [1.0] * 4, 128),
    (3, [(2, 2, 2), (130, 64, 40), (200, 180, 60)], [1.0, 2.0, 1.0], 512),
    (2, [(40, 30, 1), (700, 500, 1), (333, 801, 1)], [1.0] * 3, 128),
])
def test_order_of_the_sets_does_not_matter(ndim, dims, spacings, N):
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(N)
    images = [rng.integers(0, 200, size=d[::-1] if ndim == 3 else d[1::-1]).astype(np.uint8) for d in dims]
    p = ac.default_params(ndim, 5.0 / math.sqrt(1.5), 100.0, N=N, T=6, seed=4)
    counts, states = [], []
    for first in range(len(dims)):
        order = [(first + i) % len(dims) for i in range(len(dims))]
        volumes = [ac.ac_create_volume(images[i], spacing=(1.0, 1.0, spacings[i])) for i in order]
        sets = [ac.ac_seed(v, stride=5.0) for v in volumes]
        ac.ac_evolve_batch(sets, p)
        counts.append(ac.ac_evolve_stats(sets[0]))
        states.append({i: ac.ac_get_state(s) for i, s in zip(order, sets)})
    for c, s in zip(counts[1:], states[1:]):
        assert c == counts[0]
        for i in s:
            np.testing.assert_array_equal(s[i], states[0][i])


def test_bricks_of_the_callers_fit_a_small_first_volume():
    """Bricks too large for a staged region are cut to the first volume: such a batch is taken as
    long as that one is small, and gives what every set gives alone."""
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(3)
    dims = [(20, 12, 9), (60, 60, 60), (44, 50, 41)]
    p = ac.EvolveParams(N=33, T=4, eps0=0.02, Rmin=0.5, Rmax=6.0, seed=5, brick=(60, 60, 60))
    volumes = [ac.ac_create_volume(rng.random(d[::-1]).astype(np.float32)) for d in dims]
    sets = [ac.ac_seed(v, stride=5.0) for v in volumes]
    ac.ac_evolve_batch(sets, p)
    for c, v in zip(sets, volumes):
        alone = ac.ac_seed(v, stride=5.0)
        ac.ac_evolve(alone, ac.EvolveParams(N=33, T=4, eps0=0.02, Rmin=0.5, Rmax=6.0, seed=5))
        np.testing.assert_array_equal(ac.ac_get_state(c), ac.ac_get_state(alone))
    with pytest.raises(ac.ACError):
        ac.ac_evolve_batch(sets[::-1], p)
