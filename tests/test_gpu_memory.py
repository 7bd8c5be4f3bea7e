"""What a context holds goes back to the library's pool when it is destroyed, and
skim_release_memory hands it to the device: after a round of create, build, seeds
and queries as much device memory is free as before it."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _free():
    import torch

    import paper_1408_6282_gb300 as pkg
    torch.cuda.synchronize()
    pkg.skim_release_memory()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("build_first", [True, False])
def test_build_and_seeds_leave_no_memory_behind(build_first):
    import paper_1408_6282_gb300 as pkg
    n = 1 << 23  # arrays per node of 32 MB
    g = synth.rmat(14, 8, 3)

    def once():
        with pkg.Skim(n, g.src, g.dst, 1, 4, 0, 0.3, 1, 2, 3) as sk:
            if build_first:
                sk.build_sketches()
            sk.greedy(4)
            sk.build_sketches()
            sk.query(np.arange(40, dtype=np.uint32))
    once()
    before = _free()
    once()
    assert _free() >= before - (1 << 20)


def test_a_refused_allocation_costs_one_call(monkeypatch):
    """Every device allocation of a context refused in turn (SKIM_REFUSE_ALLOC): the call
    that wanted it reports SKIM_ENOMEM, the same call works when it is made again, and
    nothing stays allocated."""
    import paper_1408_6282_gb300 as pkg
    g = synth.rmat(11, 12, 8)
    ks = synth.Keys.from_seed(2)
    pb = oracle.Problem(g.n, g.src, g.dst, 8, 8, 0, 0.3, ks.coin, ks.rank, ks.prob)
    ox, oln, _ = oracle.build_sketches(pb)
    want = oracle.skim_stops(pb, 6)[:4]
    q = [np.arange(a, dtype=np.uint32) for a in (3, 2000)]
    ref = [oracle.union_estimate(ox, oln, 8, s) for s in q]

    def create():
        return pkg.Skim(g.n, g.src, g.dst, 8, 8, 0, 0.3, ks.coin, ks.rank, ks.prob)

    create().close()
    before = _free()
    refused = []
    for at in range(1, 111):
        monkeypatch.setenv("SKIM_REFUSE_ALLOC", str(at))
        hit = []

        def twice(f, between=lambda: None):
            try:
                return f()
            except pkg.SkimError as e:
                assert e.code == -2 and not hit
                hit.append(f)
                monkeypatch.delenv("SKIM_REFUSE_ALLOC")
                between()
                return f()

        with twice(create) as sk:
            for rows in (True, False):
                sk.set_live_rows(rows)
                twice(sk.build_sketches)
                x, ln = sk.sketches()
                assert np.array_equal(ln, oln) and np.array_equal(x, ox), at
                for a, b in zip(twice(lambda: sk.greedy_stops(6), sk.greedy_reset), want):
                    assert np.array_equal(a, b), at
            for a, b in zip(twice(lambda: sk.query_batch(q)), ref):
                assert abs(a - b) <= 1e-12 * b
            twice(sk.node_estimates)
        refused.append(len(hit))
    assert sum(refused) >= 60 and not any(refused[-5:])  # past the last allocation
    assert _free() >= before - (1 << 20)


def test_a_build_does_without_workspace_it_can_spare(monkeypatch):
    """Contraction is a shortcut: a refused allocation of its workspace leaves the build
    as it would be without it, so a graph with components wants no more than one without."""
    import paper_1408_6282_gb300 as pkg
    g = synth.rmat(11, 12, 8)
    refused = {}
    for p in (1e-6, 0.3):
        pb = oracle.Problem(g.n, g.src, g.dst, 8, 8, 0, p, 5, 6, 7)
        ox, oln, _ = oracle.build_sketches(pb)
        refused[p] = 0
        for at in range(30, 80):
            monkeypatch.setenv("SKIM_REFUSE_ALLOC", str(at))
            try:
                sk = pkg.Skim(g.n, g.src, g.dst, 8, 8, 0, p, 5, 6, 7)
            except pkg.SkimError as e:
                assert e.code == -2
                continue
            with sk:
                try:
                    sk.build_sketches()
                except pkg.SkimError as e:
                    assert e.code == -2
                    refused[p] += 1
                    sk.build_sketches()
                x, ln = sk.sketches()
                assert np.array_equal(ln, oln) and np.array_equal(x, ox), (p, at)
    assert refused[0.3] == refused[1e-6] > 5
