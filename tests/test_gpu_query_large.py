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
