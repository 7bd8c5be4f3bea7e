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
