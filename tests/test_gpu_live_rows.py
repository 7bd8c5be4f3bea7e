"""Stored instances (graph.cu) at the row sizes where they can go wrong: none, one
tile of 32 edges, more, rows cut into pieces; one instance to 64, no coin live and
all of them.  Seeds and coverages walk the rows of out-neighbours, sketches those of
in-neighbours; both are whole numbers and must equal the oracle's."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
DEGREES = [1, 31, 32, 33, 64, 65, 2047, 2048, 2049, 4097, 6000]


def _graph(reverse):
    """Nodes with DEGREES in-neighbours (reverse: out-neighbours) among 6100 nodes, the rest without."""
    rng = np.random.default_rng(4)
    n = 6100
    a, b = [], []
    for i, d in enumerate(DEGREES):
        v = 3 + 50 * i
        a.append(rng.choice(np.setdiff1d(np.arange(n), [v]), d, replace=False).astype(np.uint32))
        b.append(np.full(d, v, np.uint32))
    src, dst = (np.concatenate(b), np.concatenate(a)) if reverse else (np.concatenate(a), np.concatenate(b))
    order = np.lexsort((dst, src))
    return n, src[order], dst[order]


@pytest.mark.parametrize("reverse", [False, True])
@pytest.mark.parametrize("l", [1, 31, 32, 33, 64])
@pytest.mark.parametrize("model,p", [(0, 1e-9), (0, 0.01), (0, 1.0), (1, 0.0)])
def test_row_sizes(model, p, l, reverse):
    import paper_1408_6282_gb300 as pkg
    n, src, dst = _graph(reverse)
    ks = synth.Keys.from_seed(21)
    k = 16
    pb = oracle.Problem(n, src, dst, l, k, model, p, ks.coin, ks.rank, ks.prob)
    ox, oln, _ = oracle.build_sketches(pb)
    seeds, cov, tau, kp, _ = oracle.skim_stops(pb, 15)
    with pkg.Skim(n, src, dst, l, k, model, p, ks.coin, ks.rank, ks.prob) as sk:
        for _ in range(2):
            sk.build_sketches()
            x, ln = sk.sketches()
            assert np.array_equal(ln, oln) and np.array_equal(x, ox)
            sk.greedy_reset()
            got = sk.greedy_stops(15)
            for a, b in zip(got, (seeds, cov, tau, kp)):
                assert np.array_equal(a, b)


@pytest.mark.parametrize("l", [1, 33, 64])
@pytest.mark.parametrize("p", [0.004, 0.7])
def test_rows_cut_into_pieces(l, p):
    """Rows of one, two and many pieces of 256 edges, and rows whose pieces are longer so that
    there are at most 1024 of them; both directions, against coins drawn in the searches."""
    import paper_1408_6282_gb300 as pkg
    degrees = [255, 256, 257, 511, 512, 513, 3001, 1024 * 256 - 1, 1024 * 256, 1024 * 256 + 1, 299_999]
    n = 300_000
    rng = np.random.default_rng(l)
    a = [rng.choice(np.setdiff1d(np.arange(n), [7 * i]), d, replace=False) for i, d in enumerate(degrees)]
    b = [np.full(d, 7 * i) for i, d in enumerate(degrees)]
    u, v = np.concatenate(a), np.concatenate(b)
    key = np.unique(np.concatenate([u << 32 | v, (v + 100) << 32 | u]).astype(np.uint64))
    src, dst = (key >> np.uint64(32)).astype(np.uint32), (key & np.uint64(0xffffffff)).astype(np.uint32)
    keep = src != dst
    with pkg.Skim(n, src[keep], dst[keep], l, 8, 0, p, 3, 4, 5) as sk:
        got = []
        for rows in (True, False):
            sk.set_live_rows(rows)
            assert sk.instance_stats()[1] == rows
            sk.build_sketches()
            got.append((*sk.sketches(), *sk.greedy_stops(5)))
        for x, y in zip(*got):
            assert np.array_equal(x, y)
