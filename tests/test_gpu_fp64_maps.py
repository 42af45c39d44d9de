"""The double-precision draw and pair map (GPU) at the ends of their ranges.

Gaussians: Box-Muller in long double on the uniforms of the oracle's Philox
words, for many pairs; -2 ln u, cosine and sine are each within 4 ulp, so R c
is within (4 / 2 + 4 + 1.5) ulp < 2e-15, relative to R. Pair maps: two SSA
steps against the oracle, where a = 2 gamma chi dt / m stays below 1/4 (the
polynomials), spreads over both sides of it, and is large throughout, with
the parity tests' 1e-11."""
import numpy as np
import pytest

from gpu_util import assert_parity

pytestmark = pytest.mark.gpu


def test_gaussians_against_long_double():
    from paper_1507_06643_gb300 import dpde
    n = 200000
    rng = np.random.default_rng(11)
    a = rng.integers(0, 1 << 27, n).astype(np.uint32)
    b = a + rng.integers(1, 1000, n).astype(np.uint32)
    step, rep = rng.integers(0, 100, n).astype(np.uint32), rng.integers(0, 4, n).astype(np.uint32)
    seed = 0x1234567890ABCDEF
    got = dpde.dpde_debug_gaussian(seed, step, rep, a, b, "fp64")
    words = dpde.dpde_debug_philox(np.stack([a, b, step, rep], 1),
                                   np.tile(np.array([seed & 0xFFFFFFFF, seed >> 32], np.uint32), (n, 1)))
    x = (words >> 8).astype(np.longdouble)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    r1, r2 = (np.sqrt(-2 * np.log((x[:, k] + 1) / 2 ** 24)) for k in (0, 2))
    t1, t2 = (2 * pi * x[:, k] / 2 ** 24 for k in (1, 3))
    ref = np.stack([r1 * np.cos(t1), r1 * np.sin(t1), r2 * np.cos(t2)], 1)
    err = np.abs(got - ref) / np.stack([r1, r1, r2], 1)
    assert err.max() < 2e-15, err.max()


@pytest.mark.parametrize("sigma,dt", [(3.0, 0.01), (5.0, 0.02), (10.0, 0.1), (0.0, 0.01)])
def test_pair_map_ranges(sigma, dt):
    specs = [(300, (4.7,) * 3, 50.0, 1.0, (1, 1, 1))]
    for _ in assert_parity(specs, "fp64", "SSA", 2, 1e-11, (3, 4, 5), sigma=sigma, dt=dt, a=1.0):
        pass
