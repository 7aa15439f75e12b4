"""The competition of ac_localize at the edges of its kernel: chains longer than one
round follows, more overlapping neighbours than a lane keeps, rows of cells at the
border of the grid, and survivor counts on both sides of the line below which the cells
come back with the counts.  The oracle's greedy visit in order of (E, k) is the result
("Results and Discussion")."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ac():
    from paper_1804_06304_gb300 import ac as m
    m.load()
    return m


def _set(ac, dims, c, R, E):
    """A contour set of the given state on an empty volume."""
    V = ac.ac_create_volume(np.zeros(dims[::-1], np.uint8))
    cR = np.column_stack([c, R]).astype(np.float32)
    C = ac.ac_seed(V, explicit=cR)
    st = ac.ac_get_state(C)
    st[4] = E
    ac.ac_set_state(C, st)
    return C, ac.ac_get_state(C)


def _check(ac, oracle, ndim, C, st, E0):
    cells = ac.ac_localize(C, E0)
    want = oracle.localize(ndim, st[:4].T.astype(np.float64), st[4].astype(np.float64), float(np.float32(E0)))
    assert list(cells["id"]) == list(want)


def test_a_long_chain(ac, oracle):
    """2,000 contours on a line, each overlapping the one before and the one after it,
    energies rising along the line: every decision waits for the one before."""
    n = 2000
    c = np.column_stack([np.arange(n) * 1.0, np.full(n, 4.0), np.full(n, 4.0)])
    C, st = _set(ac, (2048, 9, 9), c, np.full(n, 1.5), np.arange(n) - 3.0 * n)   # reach 0.79 * 1.5 = 1.19
    _check(ac, oracle, 3, C, st, 0.0)


@pytest.mark.parametrize("ndim", [2, 3])
def test_a_crowd(ac, oracle, ndim):
    """900 contours within one another's reach, equal energies among them, and a few far
    away in the corners of the volume."""
    rng = np.random.default_rng(ndim)
    dims = (60, 50, 40)[:ndim]
    c = np.zeros((908, 3))
    c[:900, :ndim] = 20.0 + rng.uniform(-1, 1, (900, ndim))
    corners = np.array([[x, y, z] for x in (0, 59) for y in (0, 49) for z in (0, 39)], float)
    c[900:] = corners if ndim == 3 else corners * [1, 1, 0]
    C, st = _set(ac, dims, c, rng.uniform(3.0, 9.0, 908), np.round(rng.uniform(-9, -1, 908), 1))
    _check(ac, oracle, ndim, C, st, -2.0)


@pytest.mark.parametrize("n", [1, 7, 9, 16384, 16385])
def test_survivor_counts(ac, oracle, n):
    rng = np.random.default_rng(n)
    dims = (150, 140, 130)
    c = rng.uniform(0, 1, (n, 3)) * (np.array(dims) - 1)
    C, st = _set(ac, dims, c, rng.uniform(2.0, 5.0, n), rng.uniform(-9, -1, n))
    _check(ac, oracle, 3, C, st, 0.0)


def test_uneven_sets_in_one_call(ac, oracle):
    rng = np.random.default_rng(3)
    sets, states = [], []
    for n in (1, 300, 2, 5000, 64):
        dims = tuple(int(v) for v in rng.integers(30, 90, 3))
        C, st = _set(ac, dims, rng.uniform(0, 1, (n, 3)) * (np.array(dims) - 1), rng.uniform(2.0, 5.0, n),
                     rng.uniform(-9, -1, n))
        sets.append(C)
        states.append(st)
    E0 = -3.0
    for cells, st in zip(ac.ac_localize_batch(sets, E0), states):
        want = oracle.localize(3, st[:4].T.astype(np.float64), st[4].astype(np.float64), E0)
        assert list(cells["id"]) == list(want)
