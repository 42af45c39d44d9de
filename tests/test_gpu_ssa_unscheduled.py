"""SSA domains that no schedule of the level form can hold (GPU): 1,200
particles in a 3.3^3 box have ~83,900 forward pairs, more than 16-bit local
indices number, so the domain runs along the colour order on one block --
once, by the deferred launches, whatever launch runs beside them. Alone,
among domains that are scheduled, and behind more of those than blocks are
resident, so that the regular launch reaches them after their schedule has
been given up. Two steps as a graph and eagerly (two streams) and profiled
(one stream), bit for bit against the class launches."""
import numpy as np
import pytest

from gpu_util import make_state

pytestmark = pytest.mark.gpu

SMALL = (1000, (6.94,) * 3, 50.0, 1.0, (1, 1, 1))
DENSE = (1200, (3.3,) * 3, 50.0, 1.0, (1, 1, 1))


@pytest.mark.parametrize("precision,small,dense", [("mixed", 0, 1), ("fp64", 0, 1), ("mixed", 3, 2), ("fp64", 3, 2),
                                                   ("mixed", 1000, 60)])
def test_unscheduled_domains_run_once(precision, small, dense):
    from paper_1507_06643_gb300 import dpde
    specs = [SMALL] * small + [DENSE] * dense
    q, p, e = make_state(specs, 5, precision == "mixed")
    reps = [dpde.make_replica(n, box, cv, br) for n, box, cv, _, br in specs]

    def run(mode, how):
        S = dpde.System(dpde.make_params(seed=9, a=5.0, precision=precision), reps)
        S.set_tuning(ssa_mode=mode)
        S.set_state(q, p, e)
        if how == "profiled":
            S.step_profiled(2, 0.002, "HYBRID")
        else:
            S.step(2, 0.002, "HYBRID", use_graph=how == "graph")
        assert S.sync() == dpde.DPDE_OK
        out = S.get_state(), S.step_launches("HYBRID")
        S.close()
        return out

    ref, classes = run(0, "graph")
    for how in ("graph", "eager", "profiled"):
        got, levels = run(2, how)
        assert levels != classes   # the level form, not the class launches again
        for a, b in zip(ref, got):
            assert np.array_equal(a, b), how
