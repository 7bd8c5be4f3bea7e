"""SKIM steps (batch.cu) where they can go wrong: the search queued behind the step
and the search that waits for it, batches of one lane word, of a word and a bit
and of all ranks, stops at a batch's last lane, searches that park work and make
the step wait, ranks that run out, a run in pieces with a sketch build between.
Seeds and coverages are whole numbers and must equal the oracle's."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
GRAPHS = {
    "rmat10": lambda: synth.rmat(10, 8, 3),
    "er2003": lambda: synth.erdos_renyi(2003, 9000, 4),
    "clique": lambda: synth.clique(70),
}


@pytest.mark.parametrize("items", [None, 128])
@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("l,k,p,bl", [(64, 16, 0.2, 0), (33, 2, 0.1, 64), (64, 5, 0.05, 65), (1, 3, 0.4, 128),
                                      (40, 64, 0.3, 1000)])
def test_steps_match_oracle(monkeypatch, name, l, k, p, bl, items):
    import paper_1408_6282_gb300 as pkg
    g = GRAPHS[name]()
    ks = synth.Keys.from_seed(l + k)
    if items:
        monkeypatch.setenv("SKIM_QUEUE_ITEMS", str(items))
    pb = oracle.Problem(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    seeds, cov, tau, kp, _ = oracle.skim_stops(pb, 40)
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob, batch_lanes=bl) as sk:
        a, b = sk.greedy(40)
        assert np.array_equal(a, seeds) and np.array_equal(b, cov)
        sk.greedy_reset()
        parts = [sk.greedy(1), sk.greedy_stops(20)[:2], sk.greedy(19)]
        assert np.array_equal(np.concatenate([x[0] for x in parts]), seeds)
        assert np.array_equal(np.concatenate([x[1] for x in parts]), cov)
        sk.greedy_reset()
        sk.greedy(7)
        sk.build_sketches()  # commits the active batch unscanned
        x, ln = sk.sketches()
        ox, oln, _ = oracle.build_sketches(pb)
        assert np.array_equal(ln, oln) and np.array_equal(x, ox)


SPARSE = {
    "rmat12": lambda: synth.rmat(12, 8, 5),
    "empty": lambda: synth.empty_graph(3001),
    "cycle": lambda: synth.cycle(4099),
}


@pytest.mark.parametrize("hook", [None, ("SKIM_RECORD_ITEMS", "2048"), ("SKIM_QUEUE_ITEMS", "64")])
@pytest.mark.parametrize("name", list(SPARSE))
@pytest.mark.parametrize("l,k,p,mode", [(64, 16, 0.01, 0), (64, 64, 0.03, 0), (64, 3, 0.02, 1), (33, 32, 0.01, 0)])
def test_lanes_that_reach_their_source_only(monkeypatch, name, l, k, p, mode, hook):
    """Batches of 2^16 lanes and more: leaf lanes, and those of nodes that fill up."""
    import paper_1408_6282_gb300 as pkg
    g = SPARSE[name]()
    ks = synth.Keys.from_seed(l + k)
    if hook:
        monkeypatch.setenv(*hook)
    pb = oracle.Problem(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    seeds, cov, tau, kp, _ = oracle.skim_stops(pb, 60, rank_mode=mode)
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob, rank_mode=mode) as sk:
        got = sk.greedy_stops(60)
        for a, b in zip(got, (seeds, cov, tau, kp)):
            assert np.array_equal(a, b)
        sk.greedy_reset()
        a, b = sk.greedy(60)
        assert np.array_equal(a, seeds) and np.array_equal(b, cov)


@pytest.mark.parametrize("bl", [3071, 3072, 3073, 6200])
@pytest.mark.parametrize("name", ["rmat10", "clique"])
def test_commits_of_few_and_many_lanes(name, bl):
    """Lanes counted in a block's shared memory up to 3072 of a commit, globally above."""
    import paper_1408_6282_gb300 as pkg
    g = GRAPHS[name]()
    ks = synth.Keys.from_seed(bl)
    l, k, p = 64, 64, 0.02
    pb = oracle.Problem(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    seeds, cov, tau, kp, _ = oracle.skim_stops(pb, 30)
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob, batch_lanes=bl) as sk:
        for a, b in zip(sk.greedy_stops(30), (seeds, cov, tau, kp)):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("name", list(GRAPHS) + ["sparse"])
@pytest.mark.parametrize("l,k,p,bl", [(64, 16, 0.2, 0), (33, 2, 0.1, 64), (64, 5, 0.01, 0), (1, 3, 0.4, 128)])
def test_builds_between_seeds_lose_no_stop(name, l, k, p, bl):
    """Sketches built between two calls: the sequence goes on where it stopped, with the
    ranks of the batch that was active then."""
    import paper_1408_6282_gb300 as pkg
    g = synth.rmat(12, 8, 5) if name == "sparse" else GRAPHS[name]()
    ks = synth.Keys.from_seed(l + k)
    pb = oracle.Problem(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    seeds, cov, tau, kp, _ = oracle.skim_stops(pb, 40)
    with pkg.Skim(g.n, g.src, g.dst, l, k, 0, p, ks.coin, ks.rank, ks.prob, batch_lanes=bl) as sk:
        got = []
        for c in (7, 1, 2, 30):
            got.append(sk.greedy_stops(c))
            sk.build_sketches()
        for q, want in enumerate((seeds, cov, tau, kp)):
            assert np.array_equal(np.concatenate([x[q] for x in got]), want)


def test_coin_batches_keep_to_their_lanes():
    """With coins drawn in the searches no batch has more than 2M lanes (over stored rows
    16M, where most have no record); ranks that run out."""
    import paper_1408_6282_gb300 as pkg
    g = synth.empty_graph(300_000)
    with pkg.Skim(g.n, g.src, g.dst, 64, 255, 0, 0.1, 1, 2, 3) as sk:
        for rows, most in ((True, 1 << 24), (False, 1 << 21)):
            sk.set_live_rows(rows)
            seeds, cov = sk.greedy(3)
            assert seeds.tolist() == [0, 1, 2] and cov.tolist() == [64] * 3
            st = sk.stats()
            assert st["ranks"] == 64 * g.n and st["batches"] >= -(-st["ranks"] // most)


@pytest.mark.parametrize("scale,p,k", [(16, 0.1, 16), (17, 0.03, 32)])
def test_batches_too_large_for_their_stops(scale, p, k):
    """Batches of a million records and more whose stops follow closely are left for smaller
    ones: the same sequence as with batches that are small from the start."""
    import paper_1408_6282_gb300 as pkg
    g = synth.rmat(scale, 16, 3)
    got = []
    for bl in (0, 1 << 15):
        with pkg.Skim(g.n, g.src, g.dst, 64, k, 0, p, 5, 6, 7, batch_lanes=bl) as sk:
            parts = [sk.greedy_stops(c) for c in (300, 1, 99)]
            got.append([np.concatenate([x[q] for x in parts]) for q in range(4)])
    for a, b in zip(*got):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("k", [20, 40, 100])
@pytest.mark.parametrize("p", [0.02, 0.06, 0.2])
def test_records_of_a_node_in_order(k, p):
    """Nodes with up to 8, 32, 64, 128 and more records in a batch."""
    import paper_1408_6282_gb300 as pkg
    g = synth.rmat(11, 12, 9)
    pb = oracle.Problem(g.n, g.src, g.dst, 64, k, 0, p, 7, 8, 9)
    want = oracle.skim_stops(pb, 80)
    with pkg.Skim(g.n, g.src, g.dst, 64, k, 0, p, 7, 8, 9) as sk:
        for a, b in zip(sk.greedy_stops(80), want):
            assert np.array_equal(a, b)
