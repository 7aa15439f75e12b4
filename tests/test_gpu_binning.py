"""Contours grouped by brick ahead of the brick kernel: the one-CTA form, the
three-launch form and the sorted list for a few contours in many bricks give the
brick kernel the same contours, at the edges of their ranges ("Parallel Contour
Evaluation").  The plain path visits contours without any grouping and gives the
same bits, so every form is compared with it; the path counters must add up to the
contour-iterations of the launch alone (a form starts them from zero)."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ac():
    from paper_1804_06304_gb300 import ac as m
    m.load()
    return m


def _seeds(n, dims, rng):
    c = [rng.uniform(0, d - 1, n) for d in dims] + [np.zeros(n)] * (3 - len(dims))
    return np.column_stack(c + [rng.uniform(1.0, 2.5, n)]).astype(np.float32)


def _run(ac, V, seeds, p):
    C = ac.ac_seed(V, explicit=seeds)
    for _ in range(2):   # the second call continues on the first one's state
        ac.ac_evolve(C, p)
        assert sum(ac.ac_evolve_stats(C)) == len(seeds) * p.T
    return ac.ac_get_state(C)


# contours around the one-CTA form's 12,288; bricks around its 8,192; one contour;
# a few contours in 262,144 bricks (sorted list)
@pytest.mark.parametrize("n,dims,brick", [
    (1, (64, 64, 64), (32, 32, 32)),
    (12288, (64, 64, 64), (16, 16, 16)),
    (12289, (64, 64, 64), (16, 16, 16)),
    (3000, (64, 64, 128), (4, 4, 4)),
    (3000, (64, 64, 132), (4, 4, 4)),
    (700, (128, 128, 128), (2, 2, 2)),
    (2500, (400, 300), (7, 5, 0)),
])
def test_forms_give_the_plain_paths_bits(ac, n, dims, brick):
    rng = np.random.default_rng(n)
    vol = rng.integers(0, 255, size=dims[::-1], dtype=np.uint8)
    V = ac.ac_create_volume(vol)
    p = ac.EvolveParams(N=32, T=2, eps0=0.02, Rmin=0.5, Rmax=4.0, seed=5, brick=brick, halo_factor=1.0)
    seeds = _seeds(n, dims, rng)
    np.testing.assert_array_equal(_run(ac, V, seeds, p), _run(ac, V, seeds, dataclasses.replace(p, path=1)))


def test_many_sets_share_one_grouping(ac):
    """Forty sets, empty ones among them, in one launch: each gives what it gives alone."""
    rng = np.random.default_rng(9)
    p = ac.EvolveParams(N=32, T=2, eps0=0.02, Rmin=0.5, Rmax=4.0, seed=5)
    sets, want = [], []
    for i in range(40):
        dims = tuple(int(v) for v in rng.integers(8, 40, 3))
        V = ac.ac_create_volume(rng.integers(0, 255, size=dims[::-1], dtype=np.uint8))
        seeds = _seeds(0 if i % 7 == 3 else int(rng.integers(1, 900)), dims, rng)
        sets.append(ac.ac_seed(V, explicit=seeds))
        alone = ac.ac_seed(V, explicit=seeds)
        ac.ac_evolve(alone, p)
        want.append(ac.ac_get_state(alone))
    ac.ac_evolve_batch(sets, p)
    for c, w in zip(sets, want):
        np.testing.assert_array_equal(ac.ac_get_state(c), w)


def test_static_entry_takes_the_sorted_list_when_ranges_do_not_fit(ac):
    """3.4 million bricks: the ranges (27 MB) exceed the fixed array; 950,000 contours keep
    the bricks below the point where the list would be sorted anyway."""
    import torch
    rng = np.random.default_rng(2)
    n, dims = 950_000, (304, 304, 304)
    V = torch.randint(0, 255, dims[::-1], dtype=torch.uint8, device="cuda")
    state = np.zeros((5, n), np.float32)
    state[:4] = _seeds(n, dims, rng).T
    p = ac.EvolveParams(N=32, T=1, eps0=0.02, Rmin=0.5, Rmax=4.0, seed=5, brick=(2, 2, 2), halo_factor=1.0,
                        update_last=1)
    out = []
    for path in (0, 1):
        s = torch.as_tensor(state, device="cuda").clone()
        ac.ac_evolve_static(V, s, dataclasses.replace(p, path=path), r0=2.5, stride=3.0)
        out.append(s.cpu().numpy())
    np.testing.assert_array_equal(out[0], out[1])
