"""Queries at the sizes where their kernels change: seeds as kernel arguments and
in memory, one block, clusters, parts and the table in memory, tables at their fill limits, seeds given
twice, no seeds.  Alone and in a batch the same bits; within 1e-12 of the
oracle's sum in double."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
REL = 1e-12


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("k", [2, 16, 64, 255])
def test_sizes_around_the_limits(k, mode):
    import paper_1408_6282_gb300 as pkg
    g = synth.erdos_renyi(3001, 15000, 41)
    ks = synth.Keys.from_seed(41)
    l, p = 16, 0.15
    pb = oracle.Problem(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    ox, oln, _ = oracle.build_sketches(pb, rank_mode=mode)
    limits = [1500 // (k - 1), 2700 // (k - 1), 8000 // (k - 1), 124800 // (k - 1), 60, 960, 8000]
    sizes = sorted({s for x in limits for s in (x - 1, x, x + 1) if 0 <= s <= 9000} | {0, 1, 31, 32, 33})
    rng = np.random.default_rng(k)
    sets = [rng.integers(0, g.n, s) if s > g.n else rng.choice(g.n, s, replace=False) for s in sizes]
    sets.append(np.repeat(sets[-1][:40], 3))
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob, rank_mode=mode) as sk:
        sk.build_sketches()
        batch = sk.query_batch(sets)
        for s, b in zip(sets, batch):
            a = sk.query(s)
            assert a == b
            ref = oracle.union_estimate(ox, oln, l, s, rank_mode=mode)
            assert abs(a - ref) <= REL * abs(ref)


@pytest.mark.parametrize("large", [1, 8, 9, 16, 17, 64, 65])
@pytest.mark.parametrize("k,seeds", [(16, 181), (16, 2000), (64, 400), (64, 600), (64, 2200)])
def test_calls_with_some_larger_queries(large, k, seeds):
    """Clusters of 16 and of 4, parts; small queries and empty ones beside them."""
    import paper_1408_6282_gb300 as pkg
    g = synth.erdos_renyi(3001, 15000, 47)
    ks = synth.Keys.from_seed(47)
    rng = np.random.default_rng(large)
    sets = [rng.choice(g.n, seeds if i < large else rng.integers(0, 30), replace=False) for i in range(large + 21)]
    sets = [sets[i] for i in rng.permutation(len(sets))]
    with pkg.Skim(g.n, g.src, g.dst, 16, k, 0, 0.15, ks.coin, ks.rank, ks.prob) as sk:
        sk.build_sketches()
        want = [sk.query(s) for s in sets]
        for _ in range(2):
            assert np.array_equal(sk.query_batch(sets), want)


@pytest.mark.parametrize("k", [16, 64])
def test_without_clusters(monkeypatch, k):
    """A device that refuses clusters (SKIM_REFUSE_CLUSTERS): parts answer every query that
    would have taken one, alone, in a batch and served, with the same bits."""
    import paper_1408_6282_gb300 as pkg
    g = synth.erdos_renyi(3001, 15000, 53)
    rng = np.random.default_rng(k)
    sets = [rng.choice(g.n, s, replace=False).astype(np.uint32) for s in (0, 5, 95, 110, 200, 700, 1000, 3000)]
    sets.append(np.tile(sets[-1], 2))
    got = []
    for refuse in (False, True):
        if refuse:
            monkeypatch.setenv("SKIM_REFUSE_CLUSTERS", "1")
        with pkg.Skim(g.n, g.src, g.dst, 16, k, 0, 0.15, 3, 4, 5) as sk:
            sk.build_sketches()
            alone = [sk.query(s) for s in sets]
            few = [sk.query_batch(sets[i:i + 2]) for i in range(len(sets) - 1)]
            with sk.server(max_inflight=8, scratch_slots=1 << 21, streams=2) as srv:
                served = [srv.wait(t, 60000) for t in [srv.submit(s) for s in sets]]
            assert served == alone and all(np.array_equal(f, alone[i:i + 2]) for i, f in enumerate(few))
            got.append(alone)
    assert got[0] == got[1]


@pytest.mark.parametrize("large,small,launches", [(0, 152, 1), (0, 153, 1), (0, 456, 1), (0, 457, 1), (1, 207, 1),
                                                  (1, 208, 2), (8, 200, 1), (8, 201, 2), (20, 304, 1), (20, 305, 2),
                                                  (70, 300, 2), (1, 5000, 2)])
def test_calls_with_many_small_queries(large, small, launches):
    """Blocks of 1024, 512 and 256 threads for small queries; beside larger ones in their
    launch while they are few, else in one of their own."""
    import paper_1408_6282_gb300 as pkg
    g = synth.erdos_renyi(3001, 15000, 59)
    rng = np.random.default_rng(large + small)
    sets = [rng.choice(g.n, 70 if i < large else rng.integers(0, 43), replace=False).astype(np.uint32)
            for i in range(large + small)]
    sets = [sets[i] for i in rng.permutation(len(sets))]
    with pkg.Skim(g.n, g.src, g.dst, 16, 64, 0, 0.15, 3, 4, 5) as sk:
        sk.build_sketches()
        want = [sk.query(s) for s in sets]
        sk.query_batch(sets)
        before = pkg.skim_kernel_launches()
        assert np.array_equal(sk.query_batch(sets), want)
        assert pkg.skim_kernel_launches() - before == launches


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 9, 10, 17, 18, 33, 34])
def test_rows_read_by_a_warp_at_a_step(k, mode):
    """Rows of 1, 2, up to 4, 8 and 16 ranks share a warp's step, longer ones have it alone;
    sketches that are not full, counts of seeds that leave lanes over."""
    import paper_1408_6282_gb300 as pkg
    g = synth.erdos_renyi(3001, 5000, 67)
    ks = synth.Keys.from_seed(67)
    l, p = 16, 0.3
    pb = oracle.Problem(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    ox, oln, _ = oracle.build_sketches(pb, rank_mode=mode)
    rng = np.random.default_rng(k)
    sets = [rng.choice(g.n, s, replace=False) for s in (1, 2, 7, 31, 33, 65, 500, 1023, 3001)]
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob, rank_mode=mode) as sk:
        sk.build_sketches()
        few, many = sk.query_batch(sets), sk.query_batch(sets * 20)
        assert np.array_equal(np.tile(few, 20), many)
        for s, b in zip(sets, few):
            assert sk.query(s) == b
            ref = oracle.union_estimate(ox, oln, l, s, rank_mode=mode)
            assert abs(b - ref) <= REL * abs(ref)
