"""The sketch build over materialised rows (build.cu) at the sizes where it can
go wrong: row capacities (k at 64 and 255, fewer and more ranks than k), one
instance and 64, components contracted in one graph and in many (uniform ranks
and positions), walks that do not fit their scratch, tiny record and task
tables, node ids past the 32-bit keys of the warps' reached sets.  Sketches are
whole numbers and must equal the oracle's, or the build with coins drawn in the
searches where the oracle would take too long."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _check(n, src, dst, l, k, model, p, mode=0, bl=0, seed=31):
    import paper_1408_6282_gb300 as pkg
    ks = synth.Keys.from_seed(seed)
    pb = oracle.Problem(n, src, dst, l, k, model, p, ks.coin, ks.rank, ks.prob)
    ox, oln, _ = oracle.build_sketches(pb, rank_mode=mode)
    with pkg.Skim(n, src, dst, l, k, model, p, ks.coin, ks.rank, ks.prob, batch_lanes=bl, rank_mode=mode) as sk:
        for _ in range(2):  # a context builds again from its own leftovers
            sk.build_sketches()
            x, ln = sk.sketches()
            assert np.array_equal(ln, oln) and np.array_equal(x, ox)


GRAPHS = {
    "rmat12": lambda: synth.rmat(12, 16, 5),
    "er5000": lambda: synth.erdos_renyi(5003, 40009, 6),
    "cycle": lambda: synth.cycle(700),
    "clique": lambda: synth.clique(90),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("l,k,model,p", [(64, 64, 0, 0.1), (64, 65, 1, 0.0), (33, 255, 0, 0.3), (1, 64, 0, 0.5),
                                         (64, 2, 2, 0.0), (5, 7, 0, 1.0)])
@pytest.mark.parametrize("mode,bl", [(0, 0), (1, 0), (0, 100)])
def test_rows_match_oracle(name, l, k, model, p, mode, bl):
    g = GRAPHS[name]()
    _check(g.n, g.src, g.dst, l, k, model, p, mode, bl)


@pytest.mark.parametrize("hook,value", [("SKIM_QUEUE_ITEMS", "600"), ("SKIM_RECORD_ITEMS", "4096")])
@pytest.mark.parametrize("name", ["rmat12", "cycle"])
def test_small_scratch(monkeypatch, hook, value, name):
    monkeypatch.setenv(hook, value)
    g = GRAPHS[name]()
    _check(g.n, g.src, g.dst, 16, 16, 0, 0.2)


@pytest.mark.parametrize("count", [2, 70])
def test_components_of_many_graphs(count):
    """A component, hit lists and pivots per graph; sizes from one node up."""
    import paper_1408_6282_gb300 as pkg
    gs = [synth.empty_graph(1), synth.clique(40)] + [synth.rmat(6 + g % 4, 12, 900 + g) for g in range(count)]
    l, k = 64, 32
    keys = [synth.Keys.from_seed(200 + g) for g in range(len(gs))]
    models = [g % 3 for g in range(len(gs))]
    with pkg.Skim.batch([(g.n, g.src, g.dst) for g in gs], l, k, models, [0.3] * len(gs), [q.coin for q in keys],
                        [q.rank for q in keys], [q.prob for q in keys]) as sk:
        sk.build_sketches()
        x, ln = sk.sketches()
        for g, m, q, o in zip(gs, models, keys, sk.offsets):
            pb = oracle.Problem(g.n, g.src, g.dst, l, k, m, 0.3, q.coin, q.rank, q.prob)
            ox, oln, _ = oracle.build_sketches(pb)
            assert np.array_equal(ln[o:o + g.n], oln) and np.array_equal(x[o:o + g.n], ox)


def test_node_ids_past_24_bits():
    """2^24 + 9 nodes with edges among the highest ids (64-bit reached-set keys),
    against the build with coins drawn in the searches."""
    import paper_1408_6282_gb300 as pkg
    n = (1 << 24) + 9
    g = synth.rmat(15, 8, 77)
    src, dst = g.src + np.uint32(n - g.n), g.dst + np.uint32(n - g.n)
    with pkg.Skim(n, src, dst, 2, 8, 0, 0.25, 3, 4, 5) as sk:
        sk.build_sketches()
        x, ln = sk.sketches()
        sk.set_live_rows(False)
        sk.build_sketches()
        y, lm = sk.sketches()
        assert np.array_equal(ln, lm) and np.array_equal(x, y)


@pytest.mark.parametrize("n", [510, 511, 512, 513, 514, 1500])
@pytest.mark.parametrize("width", [1, 31, 32, 33])
def test_long_narrow_components(n, width):
    """Rings of n layers: walks of more levels than a narrow component is followed."""
    a = np.arange(n * width, dtype=np.uint32)
    layer, pos = a // width, a % width
    src = np.concatenate([a, a])
    dst = np.concatenate([((layer + 1) % n) * width + pos, ((layer + 1) % n) * width + (pos + 1) % width])
    key = np.unique(src.astype(np.uint64) << np.uint64(32) | dst.astype(np.uint64))
    _check(n * width, (key >> np.uint64(32)).astype(np.uint32), (key & np.uint64(0xffffffff)).astype(np.uint32), 3, 8, 0, 1.0)


@pytest.mark.parametrize("hubs,spokes", [(3, 640), (3, 735), (40, 1500), (1, 9000)])
def test_searches_deferred_inside_a_long_row(hubs, spokes):
    """Rows swept by a warp whose entries overflow the warp's reached set on the way
    (704 of 1024 slots): the whole warp leaves the row at the same entry.  Few lanes
    start at a hub, so batches stay with the warps' own searches."""
    n = hubs * (spokes + 1) + 12000
    h = np.arange(hubs, dtype=np.uint32)
    src = (np.arange(hubs * spokes, dtype=np.uint32) + np.uint32(hubs))
    dst = np.repeat(h, spokes)
    order = np.lexsort((dst, src))
    _check(n, src[order], dst[order], 16, 64, 0, 1.0)
    _check(n, src[order], dst[order], 16, 64, 0, 0.9, mode=1)


def test_components_of_more_graphs_than_a_grid_dimension():
    """66000 rings of 80 nodes, contracted: a list per graph and instance, against the
    build with coins drawn in the searches."""
    import paper_1408_6282_gb300 as pkg
    count, size = 66000, 80
    a = np.arange(size, dtype=np.uint32)
    ring = (size, a, np.roll(a, -1))
    keys = [synth.Keys.from_seed(g % 977) for g in range(count)]
    with pkg.Skim.batch([ring] * count, 2, 3, [0] * count, [1.0] * count, [q.coin for q in keys],
                        [q.rank + g for g, q in enumerate(keys)], [q.prob for q in keys]) as sk:
        sk.build_sketches()
        x, ln = sk.sketches()
        sk.set_live_rows(False)
        sk.build_sketches()
        y, lm = sk.sketches()
        assert np.array_equal(ln, lm) and np.array_equal(x, y)
        assert np.all(ln == 3)


@pytest.mark.parametrize("l,k,p", [(1, 16, 0.1), (1, 64, 0.3), (4, 16, 0.1), (4, 32, 0.1), (2, 64, 0.05)])
def test_few_instances(l, k, p):
    """Where the first batch gives components all their ranks, and where it does not."""
    for scale in (10, 13):
        g = synth.rmat(scale, 16, 3)
        _check(g.n, g.src, g.dst, l, k, 0, p)


@pytest.mark.parametrize("records", [None, "70000", "6000"])
@pytest.mark.parametrize("l,k,p", [(1, 255, 0.15), (16, 128, 0.15), (1, 16, 0.4)])
def test_batches_of_many_visits_per_entry(monkeypatch, records, l, k, p):
    """Later batches with a record per table entry, appended in parts of as many lanes as
    the record table holds, by count and (a small table, that of 64 lanes) by the most
    there can be."""
    if records:
        monkeypatch.setenv("SKIM_RECORD_ITEMS", records)
    g = synth.erdos_renyi(5003, 40009, 6)
    _check(g.n, g.src, g.dst, l, k, 0, p)
