"""Large queries where their form changes: the table in global memory by ranks, with
long rows later, and by seeds for a query alone with short rows; clusters of one
and of two rounds.  Alone and beside another query the same bits; within 1e-12 of the
oracle's sum in double."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,seeds", [(2, 24999), (2, 25001), (3, 60000), (8, 25001), (9, 50001), (16, 60000),
                                     (33, 34299), (33, 34301), (64, 17422), (64, 20000), (64, 23809), (64, 23810)])
def test_large_queries(k, seeds):
    import paper_1408_6282_gb300 as pkg
    g = synth.erdos_renyi(70001, 140000, 61)
    ks = synth.Keys.from_seed(61)
    l, p = 40, 0.3
    pb = oracle.Problem(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    rng = np.random.default_rng(k + seeds)
    s = rng.choice(g.n, seeds, replace=False).astype(np.uint32)
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob) as sk:
        sk.build_sketches()
        x, ln = sk.sketches()
        a = sk.query(s)
        assert np.array_equal(sk.query_batch([s, s[:5]]), [a, sk.query(s[:5])])
        assert sk.query(s) == a
        ref = oracle.union_estimate(x, ln, l, s)
        assert abs(a - ref) <= 1e-12 * ref


@pytest.mark.parametrize("large", [1, 7, 13, 16])
@pytest.mark.parametrize("small", [4, 14, 100, 150, 300])
def test_small_queries_beside_large_ones(large, small):
    """In one launch with the clusters of 16 and in one of their own: the same bits as alone."""
    import paper_1408_6282_gb300 as pkg
    g = synth.erdos_renyi(5003, 20000, 62)
    ks = synth.Keys.from_seed(62)
    l, k, p = 40, 64, 0.3
    rng = np.random.default_rng(100 * large + small)
    sets = [rng.choice(g.n, s, replace=False).astype(np.uint32)
            for s in [600] + list(rng.integers(44, 1000, large - 1)) + list(rng.integers(0, 43, small))]
    sets = [sets[i] for i in rng.permutation(len(sets))]
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob) as sk:
        sk.build_sketches()
        assert np.array_equal(sk.query_batch(sets), [sk.query(s) for s in sets])
