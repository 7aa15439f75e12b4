"""Localization of many sets in one call: the rounds take the sets in turn, their first
survivors before what larger sets have beyond them, and find a survivor's set by a search
of 32 sets at a time.  Every set gets the cells that it gets alone, at set counts around
the powers of 32, with empty sets, sets without survivors, sets around a block's eight
survivors, and sets much larger than the others."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# the rounds take the sets in turn from 19,456 survivors in all
@pytest.mark.parametrize("n_sets,largest", [(2, 6000), (31, 6000), (32, 6000), (33, 6000), (70, 6000), (1023, 6000),
                                            (1025, 6000), (2, 40000), (31, 40000), (33, 40000), (70, 40000)])
def test_sets_of_one_call_give_what_each_gives_alone(n_sets, largest):
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(n_sets)
    V = ac.ac_create_volume(np.zeros((20, 40, 60), np.uint8))
    sizes = rng.choice([0, 1, 7, 8, 9, 40, 300], n_sets)
    sizes[rng.integers(n_sets, size=2)] = [largest, largest // 4]   # far above the mean: beyond the heads
    sets = []
    for n in sizes:
        c = rng.uniform(0, 1, (n, 3)) * [59, 39, 19]
        s = ac.ac_seed(V, explicit=np.column_stack([c, rng.uniform(1.0, 5.0, n)]).astype(np.float32))
        state = ac.ac_get_state(s)
        state[4] = rng.uniform(-1.0, 0.3, n) if rng.random() < 0.9 else 1.0
        ac.ac_set_state(s, state)
        sets.append(s)
    for got, s in zip(ac.ac_localize_batch(sets, 0.0), sets):
        np.testing.assert_array_equal(got, ac.ac_localize(s, 0.0))


def test_neighbour_grids_of_2_31_minus_1_cells():
    """The most cells one call takes (their starts are one more than an int counts): 31 sets of
    512 x 512 x 256 cells and one of 3 x 2731 x 8191, by spacings wide against the radii."""
    from paper_1804_06304_gb300 import ac
    cell = float(np.float32(0.79370052598409973738)) * 1.0001
    sets, cells = [], 0
    for shape in [(512, 512, 256)] * 31 + [(3, 2731, 8191)]:
        sp = tuple(float(np.float32((k - 0.5) * cell)) for k in shape)
        V = ac.ac_create_volume(np.zeros((2, 2, 2), np.uint8), spacing=sp)
        # two apart, one that overlaps the first, one that overlaps the last
        c = np.array([[0, 0, 0], sp, [0.5, 0, 0], sp], np.float32) - [[0, 0, 0], [0, 0, 0], [0, 0, 0], [0.25, 0, 0]]
        s = ac.ac_seed(V, explicit=np.column_stack([c, np.ones(4)]).astype(np.float32))
        state = ac.ac_get_state(s)
        state[4] = [-3.0, -1.0, -2.0, -4.0]
        ac.ac_set_state(s, state)
        cells += int(np.prod([int(np.floor(np.float32(w) / cell)) + 1 for w in sp], dtype=np.int64))
        sets.append(s)
    assert cells == 2**31 - 1
    for got in ac.ac_localize_batch(sets, 0.0):
        assert list(got["id"]) == [3, 0]
