"""Bursts of requests at the server's limits: more than fit a group, one in flight at
a time, empty seed sets, scratch for a few queries only, several submitting threads,
results taken out of order; seed sets as arrays of any integer type, lists and
mixtures.  Every estimate must be the single query's, bit for bit."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sk():
    import paper_1408_6282_gb300 as pkg
    g = synth.erdos_renyi(2003, 12000, 8)
    ks = synth.Keys.from_seed(8)
    with pkg.Skim(g.n, g.src, g.dst, 8, 16, 0, 0.2, ks.coin, ks.rank, ks.prob) as s:
        s.build_sketches()
        yield s


def _sets(n, count):
    rng = np.random.default_rng(count)
    return [rng.choice(n, rng.integers(0, 40), replace=False).astype(np.uint32) for _ in range(count)]


@pytest.mark.parametrize("inflight,slots,streams", [(4096, 1 << 24, 4), (1, 1 << 14, 1), (7, 1 << 14, 3), (300, 1 << 12, 2)])
def test_burst(sk, inflight, slots, streams):
    sets = _sets(sk.n, 500)
    want = [sk.query(s) for s in sets]
    with sk.server(max_inflight=inflight, scratch_slots=slots, streams=streams) as srv:
        lat, est = srv.replay(np.zeros(len(sets)), sets)
        assert np.array_equal(est, want) and (lat > 0).all()
        got = {}

        def client(part):
            tickets = [(i, srv.submit(sets[i])) for i in range(part, len(sets), 4)]
            for i, t in reversed(tickets):
                got[i] = srv.wait(t)

        threads = [threading.Thread(target=client, args=(p,)) for p in range(4)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert [got[i] for i in range(len(sets))] == want


@pytest.mark.parametrize("kind", ["u32", "i64", "lists", "mixed", "tuple", "generator", "empty", "rows"])
def test_seed_sets_of_any_kind(sk, kind):
    base = _sets(sk.n, 9)
    base[4] = base[4][:0]
    sets = {"u32": base, "i64": [b.astype(np.int64) for b in base], "lists": [b.tolist() for b in base],
            "mixed": [b if i % 2 else b.tolist() for i, b in enumerate(base)], "tuple": tuple(base),
            "generator": base, "empty": [[], []], "rows": np.arange(60).reshape(6, 10)}[kind]
    want = [sk.query(np.asarray(s, dtype=np.uint32)) for s in sets]
    arg = (s for s in sets) if kind == "generator" else sets
    assert np.array_equal(sk.query_batch(arg), want)
    with sk.server(max_inflight=4, scratch_slots=1 << 14, streams=2) as srv:
        assert np.array_equal(srv.replay(np.zeros(len(want)), sets)[1], want)


def test_the_last_requests_do_not_wait_for_their_collection(sk):
    """A replay collects thousands of results at its end; groups still in flight are
    finished beside that.  (The last request had taken 0.2 ms where others take 0.05.)"""
    sets = _sets(sk.n, 4000)
    with sk.server(max_inflight=1024, scratch_slots=1 << 20, streams=2) as srv:
        arrive = np.arange(len(sets)) / 20000.0
        runs = [srv.replay(arrive, sets)[0] for _ in range(7)]
    assert min(r[-1] for r in runs) < 2.5 * min(np.median(r) for r in runs)
