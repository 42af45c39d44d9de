"""Handles of different sizes side by side (GPU): the limit on a kernel's
dynamic shared memory belongs to the process, so what a second, smaller handle
needs must not be what the first one gets. The first handle's results, alone
and with the second one made in between, bit for bit."""
import numpy as np
import pytest

from gpu_util import make_state

pytestmark = pytest.mark.gpu

SOFT = [(300000, (46.5,) * 3, 50.0, 1.0, (8, 8, 8))]    # the widest work tiles
SMALL = [(8000, (13.9,) * 3, 50.0, 1.0, (1, 1, 1))]     # work tiles of a cell or two, short level tables


def lennard_jones(precision):
    """Eight whole replicas of 500 particles: level tables beyond 1,023 levels."""
    from paper_1507_06643_gb300 import inputs
    q, p, e, L = inputs.fcc_state(5, 0.8095, 1.0, 50.0, 1.0, 3)
    if precision == "mixed":
        q = q.astype(np.float32).astype(np.float64)
        q = np.where(q >= L, 0.0, q)
        p = p.astype(np.float32).astype(np.float64)
    return [(len(q), (L, L, L), 50.0, 1.0, (1, 1, 1))] * 8, tuple(np.concatenate([x] * 8) for x in (q, p, e))


@pytest.mark.parametrize("graph", [True, False])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("first", ["soft_hybrid", "lj_ssa"])
def test_a_second_handle_leaves_the_first_alone(first, precision, graph):
    from paper_1507_06643_gb300 import dpde
    if first == "soft_hybrid":
        specs, scheme, dt, prm = SOFT, "HYBRID", 0.01, dict(seed=9)
        st = make_state(specs, 5, precision == "mixed")
    else:
        specs, st = lennard_jones(precision)
        scheme, dt, prm = "SSA", 0.002, dict(seed=9, r_cut=2.5, sigma=2.0, potential=1, lj_eps=1.0, lj_r=1.0)

    def system(sp, **kw):
        return dpde.System(dpde.make_params(precision=precision, **kw),
                           [dpde.make_replica(n, box, cv, br) for n, box, cv, _, br in sp])

    def run(between):
        S, other = system(specs, **prm), None
        S.set_state(*st)
        S.step(1, dt, scheme, use_graph=graph)
        if between:
            other = system(SMALL)
            S.set_state(*st)
            S.step(1, 1.5 * dt, scheme, use_graph=graph)   # (another step length: another graph)
        S.set_state(*st)
        S.step(2, 0.5 * dt, scheme, use_graph=graph)
        out = S.get_state(), S.observables()
        if other is not None:
            other.close()
        S.close()
        return out

    ref, obs = run(False)
    got, obs2 = run(True)
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
    assert obs == obs2
