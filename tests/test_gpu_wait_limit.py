"""A wait limit bounds waits without progress, not the length of a busy phase: limits
far below what a level of a large component, a step or a need pass takes leave
builds and seeds as they are."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l,model,p", [(64, 0, 0.1), (64, 1, 0.0), (8, 0, 0.3)])
def test_short_limits_do_not_end_busy_phases(l, model, p):
    import paper_1408_6282_gb300 as pkg
    g = synth.rmat(18, 16, 3)

    def run(ns):
        with pkg.Skim(g.n, g.src, g.dst, l, 64, model, p, 5, 6, 7) as sk:
            if ns:
                sk.set_wait_limit_ns(ns)
            sk.build_sketches()
            return (*sk.sketches(), *sk.greedy(20))

    for a, b in zip(run(200_000), run(0)):
        assert np.array_equal(a, b)
