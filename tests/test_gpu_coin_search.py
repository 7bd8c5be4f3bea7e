"""Reverse searches that draw their coins (no stored instances, and the IC model,
which never stores any): rows of up to, at and past the 32, 64 and 128 edges a
warp takes at a step, rows longer than a queue item takes at once, every edge live
and few, one instance per item and many.  Sketches are whole numbers and must equal
the oracle's."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
DEGREES = [1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 257, 1000, 2100]


def _graph():
    """DEGREES as in-degrees, 4 nodes of each, among 3000 nodes; a ring joins all."""
    rng = np.random.default_rng(9)
    n = 3000
    src, dst = [np.arange(n, dtype=np.uint32)], [np.roll(np.arange(n, dtype=np.uint32), 1)]
    for i, d in enumerate(DEGREES * 4):
        v = 50 * i
        u = rng.choice(np.setdiff1d(np.arange(n), [v, (v + 1) % n]), d - 1, replace=False).astype(np.uint32)
        src.append(u)
        dst.append(np.full(d - 1, v, np.uint32))
    src, dst = np.concatenate(src), np.concatenate(dst)
    order = np.lexsort((dst, src))
    return n, src[order], dst[order]


@pytest.mark.parametrize("mode,l,bl", [(2, 1, 0), (2, 1, 100), (0, 1, 0), (0, 64, 0), (1, 7, 64)])
@pytest.mark.parametrize("model,p", [(0, 0.5), (0, 0.02), (1, 0.0), (2, 0.0)])
def test_row_sizes(model, p, mode, l, bl):
    import paper_1408_6282_gb300 as pkg
    n, src, dst = _graph()
    ks = synth.Keys.from_seed(17)
    k = 33
    pb = oracle.Problem(n, src, dst, l, k, model, p, ks.coin, ks.rank, ks.prob)
    ox, oln, _ = oracle.build_ic_sketches(pb) if mode == 2 else oracle.build_sketches(pb, rank_mode=mode)
    with pkg.Skim(n, src, dst, l, k, model, p, ks.coin, ks.rank, ks.prob, batch_lanes=bl, rank_mode=mode) as sk:
        sk.set_live_rows(False)
        for _ in range(2):
            sk.build_sketches()
            x, ln = sk.sketches()
            assert np.array_equal(ln, oln) and np.array_equal(x, ox)


@pytest.mark.parametrize("p", [0.01, 0.3])
@pytest.mark.parametrize("mode,l", [(2, 1), (0, 64), (1, 64)])
def test_batches_of_few_and_many_visits(p, mode, l):
    """Batches expected to make fewer and more than 2^20 visits take different launches."""
    import paper_1408_6282_gb300 as pkg
    g = synth.rmat(11, 16, 21)
    ks = synth.Keys.from_seed(18)
    k = 40
    pb = oracle.Problem(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    ox, oln, _ = oracle.build_ic_sketches(pb) if mode == 2 else oracle.build_sketches(pb, rank_mode=mode)
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob, rank_mode=mode) as sk:
        sk.set_live_rows(False)
        for _ in range(2):
            sk.build_sketches()
            x, ln = sk.sketches()
            assert np.array_equal(ln, oln) and np.array_equal(x, ox)
        if p == 0.3:
            assert sk.stats()["rev_visits"] > 20 * 2**20 or mode != 2
        if mode != 2:
            want = oracle.skim_stops(pb, 15, rank_mode=mode)
            for a, b in zip(sk.greedy_stops(15), want):
                assert np.array_equal(a, b)


@pytest.mark.parametrize("items", [None, "600"])
@pytest.mark.parametrize("mode,l,bl", [(2, 1, 0), (2, 1, 64), (0, 64, 0)])
@pytest.mark.parametrize("degree,p", [(1, 1.0), (1, 0.99), (2, 0.6), (8, 0.2), (31, 0.05), (32, 0.05)])
def test_rows_of_one_length(degree, p, mode, l, bl, items, monkeypatch):
    """Every node has as many in-edges: from a chain of single edges, where each lane
    takes its own edge, to rows that the warp sweeps; a queue that is full at once
    (items of many lanes come back) and one that is not."""
    import paper_1408_6282_gb300 as pkg
    if items:
        monkeypatch.setenv("SKIM_QUEUE_ITEMS", items)
    n, k = 700, 33
    v = np.repeat(np.arange(n, dtype=np.uint32), degree)
    u = ((v + np.tile(21 * np.arange(degree, dtype=np.uint32) + 1, n)) % n).astype(np.uint32)
    key = np.unique(u.astype(np.uint64) << np.uint64(32) | v.astype(np.uint64))
    src, dst = (key >> np.uint64(32)).astype(np.uint32), key.astype(np.uint32)
    src, dst = src[src != dst], dst[src != dst]
    ks = synth.Keys.from_seed(23)
    pb = oracle.Problem(n, src, dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    ox, oln, _ = oracle.build_ic_sketches(pb) if mode == 2 else oracle.build_sketches(pb, rank_mode=mode)
    with pkg.Skim(n, src, dst, l, k, 0, p, ks.coin, ks.rank, ks.prob, batch_lanes=bl, rank_mode=mode) as sk:
        sk.set_live_rows(False)
        sk.build_sketches()
        x, ln = sk.sketches()
        assert np.array_equal(ln, oln) and np.array_equal(x, ox)
        if mode != 2:
            for a, b in zip(sk.greedy_stops(10), oracle.skim_stops(pb, 10, rank_mode=mode)):
                assert np.array_equal(a, b)
