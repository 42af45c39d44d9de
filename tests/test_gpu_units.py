"""FP64 in units far from one (GPU): lengths, and with them momenta, energies
and the force and noise amplitudes, scaled by a power of two, so that every
double of the run is the same up to that factor. The square of the cutoff lies
beyond the range of a float; the results are those of the unscaled run, scaled,
bit for bit."""
import numpy as np
import pytest

from gpu_util import make_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme,bricks", [("SER", (1, 1, 1)), ("HYBRID", (2, 2, 1)), ("SSA", (1, 1, 1))])
@pytest.mark.parametrize("power", [-70, 70])
def test_scaled_units(power, scheme, bricks):
    from paper_1507_06643_gb300 import dpde
    n, L = 1100, 7.3
    q, p, e = make_state([(n, (L,) * 3, 50.0, 1.0, bricks)], 5, False)

    def run(s):
        S = dpde.System(dpde.make_params(r_cut=s, a=25.0 * s, sigma=3.0 * s, seed=9, precision="fp64"),
                        [dpde.make_replica(n, (L * s,) * 3, 50.0, bricks)])
        S.set_state(q * s, p * s, e * s * s)
        S.step(2, 0.01, scheme)
        out, obs = S.get_state(), S.observables()[0]
        S.close()
        return [out[0] / s, out[1] / s, out[2] / s / s, obs["U"] / s / s, obs["Tpot_den"]]

    ref, got = run(1.0), run(2.0 ** power)
    assert ref[3] > 0.0
    for a, b in zip(ref, got):
        assert np.array_equal(a, b)
