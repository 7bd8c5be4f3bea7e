"""Residual searches with one block per instance (reach.cu) at the sizes where
they can go wrong: rows swept by the whole block, frontiers wider than the
shared buffer, frontiers that do not fit the scratch either (a small work
queue: the rest is parked and re-queued), index segments erased by the whole
block, one instance and more than 32.  Seeds, coverages, thresholds and k' are
whole numbers and must equal the oracle's."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _broom(width):
    """0 -> 1..width, i -> width + i, width + i -> 0: a long row, a wide frontier, a cycle."""
    a = np.arange(1, width + 1, dtype=np.uint32)
    src = np.concatenate([np.zeros(width, np.uint32), a, a + width])
    dst = np.concatenate([a, a + width, np.zeros(width, np.uint32)])
    order = np.lexsort((dst, src))
    return 2 * width + 1, src[order], dst[order]


@pytest.mark.parametrize("items", [None, 512])
@pytest.mark.parametrize("width", [31, 511, 512, 3000])
@pytest.mark.parametrize("l,k,p", [(1, 2, 1.0), (33, 5, 0.9), (64, 16, 0.5)])
def test_block_searches_match_oracle(monkeypatch, items, width, l, k, p):
    import paper_1408_6282_gb300 as pkg
    n, src, dst = _broom(width)
    ks = synth.Keys.from_seed(width + l)
    if items:
        monkeypatch.setenv("SKIM_QUEUE_ITEMS", str(items))
    sk = pkg.Skim(n, src, dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    pb = oracle.Problem(n, src, dst, l, k, 0, p, ks.coin, ks.rank, ks.prob)
    seeds, cov, tau, kp, _ = oracle.skim_stops(pb, 12)
    with sk:
        got = sk.greedy_stops(12)
    for a, b in zip(got, (seeds, cov, tau, kp)):
        assert np.array_equal(a, b)
