"""The SSA a warp per cell at the edges of its staging (GPU), against the level
form (whose schedule walks long rows a warp per cell), which must agree bit
for bit: cells with none, one or many rounds of entries, rows beyond 32
particles, more particles than are staged, domains that end at a brick face,
at the box's own periodic image and at a wall. Two steps each."""
import numpy as np
import pytest

from gpu_util import make_state

pytestmark = pytest.mark.gpu


def run(n, box, bricks, scheme, precision, clump, walls, mode):
    from paper_1507_06643_gb300 import dpde
    q, p, e = make_state([(n, box, 50.0, 1.0, bricks)], 5, precision == "mixed")
    if clump:   # a quarter of the particles in a corner: ~9.5 a cell, ~130 within reach
        q[:n // 4] *= clump
    S = dpde.System(dpde.make_params(seed=9, a=5.0, precision=precision),
                    [dpde.make_replica(n, box, 50.0, bricks, *walls)])
    S.set_tuning(ssa_mode=mode)
    S.set_state(q, p, e)
    S.step(2, 0.002, scheme)
    out = S.get_state()
    S.close()
    return out


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,box,bricks,scheme,clump,walls", [
    (1, (3.0, 3.0, 3.0), (1, 1, 1), "SSA", None, (0, 0.0)),
    (100, (3.0, 3.4, 4.2), (1, 1, 1), "SSA", None, (0, 0.0)),
    (1700, (7.5, 8.5, 9.5), (1, 1, 1), "SSA", None, (0, 0.0)),
    (1700, (7.5, 8.5, 9.5), (1, 1, 1), "SSA", None, (1, -0.5)),
    (1000, (6.1, 8.2, 7.3), (2, 4, 1), "HYBRID", None, (0, 0.0)),
    (2000, (9.0, 9.0, 9.0), (1, 1, 1), "SSA", 0.45, (0, 0.0)),     # a corner too dense to be staged
    (200, (3.0, 3.1, 3.2), (1, 1, 1), "SSA", None, (0, 0.0)),      # ~14 entries a row: levels by warps
    (350, (3.2, 3.2, 3.2), (1, 1, 1), "SSA", None, (0, 0.0)),      # ~22, some rows beyond 32
    (3000, (9.0, 6.2, 6.2), (3, 1, 1), "HYBRID", None, (0, 0.0)),  # ~15, in domains
    (1200, (3.3, 3.3, 3.3), (1, 1, 1), "SSA", None, (0, 0.0)),     # ~44 a cell
])
def test_cells_equal_the_levels(n, box, bricks, scheme, clump, walls, precision):
    ref = run(n, box, bricks, scheme, precision, clump, walls, 2)
    got = run(n, box, bricks, scheme, precision, clump, walls, 0)
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
