"""The path counters of a launch (fast, clamped, global gathers) do not depend on how its
contours were grouped by brick: a warp takes the slowest path any of its contours needs,
so they are the same in every run, and the same whether a brick's list was counted out or
sorted, only if every list is in index order.  Lists beyond the 128 contours that the
brick kernel orders itself: up to 1,024 (ordered by counting) and more (by bitmaps of
262,144 indices), in the one-CTA grouping and in the larger one.  The sorted list is
reached with a second set of one contour in a volume of many bricks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# `n` contours in the first `seeded` voxels of each axis of an image of `side`
@pytest.mark.parametrize("n,seeded,side,brick,other", [
    (6000, 32, 256, 8, 2800),        # one CTA: 375 contours a brick
    (12000, 32, 256, 16, 5600),      # one CTA: 3,000
    (20000, 64, 256, 8, 3200),       # 312
    (400000, 64, 512, 8, 10400),     # 6,250, indices over two bitmaps
    (20000, 64, 64, 8, 3200),        # every brick crowded
])
def test_counts_are_those_of_the_sorted_list(n, seeded, side, brick, other):
    torch = pytest.importorskip("torch")
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(n)
    V = ac.ac_create_volume(rng.integers(0, 255, size=(side, side), dtype=np.uint8))
    seeds = np.column_stack([rng.uniform(0, seeded - 1, (n, 2)), np.zeros(n), rng.uniform(0.6, 1.0, n)])
    seeds[0, 3] = 1.0
    p = ac.EvolveParams(N=64, T=2, eps0=0.0, Rmin=0.5, Rmax=1.5, seed=5, brick=(brick, brick, 0), halo_factor=1.0)
    A = ac.ac_seed(V, explicit=seeds.astype(np.float32))
    counts = []
    for _ in range(3):
        ac.ac_evolve(A, p)
        counts.append(ac.ac_evolve_stats(A))
    assert sum(counts[0]) == n * p.T and min(counts[0][:2]) > 0
    assert counts[1] == counts[0] and counts[2] == counts[0]
    assert (other // brick) ** 2 > 4 * (n + 1) + 65536
    W = ac.ac_create_volume(torch.zeros((other, other), dtype=torch.uint8, device="cuda"))
    B = ac.ac_seed(W, explicit=np.array([[other / 2, other / 2, 0.0, 1.0]], np.float32))
    ac.ac_evolve(B, p)
    alone = ac.ac_evolve_stats(B)
    ac.ac_evolve_batch([A, B], p)
    assert ac.ac_evolve_stats(A) == tuple(a + b for a, b in zip(counts[0], alone))


@pytest.mark.parametrize("n,launches", [(32768, 5), (32769, 2)])
def test_crowded_bricks_are_sorted(n, launches):
    """64 bricks: beyond a mean list of 512 contours a sort (one kernel of the library's own, beside
    the brick kernel) is cheaper than counting on so few counters (four)."""
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(n)
    V = ac.ac_create_volume(rng.integers(0, 255, size=(64, 64), dtype=np.uint8))
    seeds = np.column_stack([rng.uniform(0, 63, (n, 2)), np.zeros(n), np.ones(n)]).astype(np.float32)
    C = ac.ac_seed(V, explicit=seeds)
    before = ac.ac_kernel_launches()
    ac.ac_evolve(C, ac.EvolveParams(N=64, T=1, eps0=0.0, Rmin=0.5, Rmax=1.5, brick=(8, 8, 0)))
    assert ac.ac_kernel_launches() - before == launches


@pytest.mark.parametrize("n", [5000, 20000])
def test_counts_of_a_replayed_graph(n):
    """The grouping as part of a captured graph (its last kernel is launched ahead of the end of the
    one before): every replay counts what a plain launch counts."""
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(n)
    V = ac.ac_create_volume(rng.integers(0, 255, size=(256, 256), dtype=np.uint8))
    seeds = np.column_stack([rng.uniform(0, 40, (n, 2)), np.zeros(n), rng.uniform(0.6, 1.0, n)]).astype(np.float32)
    p = ac.EvolveParams(N=64, T=2, eps0=0.0, Rmin=0.5, Rmax=1.5, seed=5, brick=(8, 8, 0), halo_factor=1.0)
    C = ac.ac_seed(V, explicit=seeds)
    ac.ac_evolve(C, p)
    want = ac.ac_evolve_stats(C)
    plan = ac.ac_plan_create([C], p)
    for _ in range(4):
        ac.ac_plan_launch(plan, use_graph=True)
        assert ac.ac_evolve_stats(C) == want
