"""The SSA by dependency levels at the edges of its execution (GPU): domains
whose records fill none, one or many of the chunks drawn ahead, levels wider
and narrower than the applying threads. Two steps in the level form against
the class-by-class launches (the defined sequence, a thread per cell), which
must agree bit for bit."""
import numpy as np
import pytest

from gpu_util import make_state

pytestmark = pytest.mark.gpu


def run(n, box, bricks, scheme, precision, **tuning):
    from paper_1507_06643_gb300 import dpde
    specs = [(n, box, 50.0, 1.0, bricks)]
    q, p, e = make_state(specs, 5, precision == "mixed")
    S = dpde.System(dpde.make_params(seed=9, precision=precision), [dpde.make_replica(n, box, 50.0, bricks)])
    S.set_tuning(**tuning)
    S.set_state(q, p, e)
    S.step(2, 0.01, scheme)
    out = S.get_state()
    S.close()
    return out


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,edge,bricks,scheme", [
    (1, 3.0, (1, 1, 1), "SSA"), (9, 3.0, (1, 1, 1), "SSA"), (40, 3.0, (1, 1, 1), "SSA"),
    (90, 3.0, (3, 1, 1), "HYBRID"), (1100, 7.2, (2, 2, 2), "HYBRID"), (9000, 14.5, (1, 1, 1), "SSA")])
def test_level_form_equals_the_sequence(n, edge, bricks, scheme, precision):
    ref = run(n, (edge,) * 3, bricks, scheme, precision, ssa_mode=0)
    for block in (32, 64, 128):
        got = run(n, (edge,) * 3, bricks, scheme, precision, ssa_mode=2, ssa_block=block)
        for a, b in zip(ref, got):
            assert np.array_equal(a, b), block
