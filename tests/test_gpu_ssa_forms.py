"""The forms of the SSA against one another where each can go wrong (GPU), with
the launch counts that tell which form ran: cells of more than 32 particles in
a warp's rows, a domain of hundreds of chunks whose state exceeds shared
memory, classes of more than 32 cells per SM (a thread per cell), sparse
systems (cells too empty for a warp). The reference is the persistent launch
(ssa_mode 3: each cell's chain by one thread, a grid barrier between classes).
Two steps, bit for bit."""
import numpy as np
import pytest

from gpu_util import make_state

pytestmark = pytest.mark.gpu

CASES = {
    # ~44 particles a cell: the warp's rows in two rounds
    "full_cells": (1200, (3.3, 3.3, 3.3), (1, 1, 1), "SSA", 0.002, False),
    # one domain of 9,000: ~56,000 records, 440 chunks
    "one_domain": (9000, (14.5, 14.5, 14.5), (1, 1, 1), "HYBRID", 0.01, True),
    # 110,592 cells in 18 classes of 6,144, on at most 152 SMs
    "large_classes": (331776, (48.1, 48.1, 48.1), (8, 8, 8), "HYBRID", 0.01, True),
    "large_replica": (400000, (52.3, 51.2, 50.4), (1, 1, 1), "SSA", 0.01, False),
    "sparse": (3000, (24.7, 25.2, 23.9), (1, 1, 1), "SSA", 0.01, True),
    "sparse_domains": (3000, (24.7, 25.2, 23.9), (2, 3, 2), "HYBRID", 0.01, True),
}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", list(CASES))
def test_forms_agree_with_the_persistent_launch(case, precision):
    from paper_1507_06643_gb300 import dpde
    n, box, bricks, scheme, dt, levels = CASES[case]
    st = make_state([(n, box, 50.0, 1.0, bricks)], 5, precision == "mixed")
    S = dpde.System(dpde.make_params(seed=9, a=5.0, precision=precision), [dpde.make_replica(n, box, 50.0, bricks)])
    out, launches = {}, {}
    for mode in (3, 0, 2):
        S.set_tuning(ssa_mode=mode)
        S.set_state(*st)
        S.step(2, dt, scheme)
        assert S.sync() == dpde.DPDE_OK
        out[mode], launches[mode] = S.get_state(), S.step_launches(scheme)
    S.close()
    assert launches[3] < launches[0]                   # one launch for all classes
    assert (launches[2] != launches[0]) == levels      # the level form, or the class launches again
    for mode in (0, 2):
        for a, b in zip(out[3], out[mode]):
            assert np.array_equal(a, b), mode
