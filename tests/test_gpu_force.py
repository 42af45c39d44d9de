"""Parity of the tiled force pass at the edges of its tiles and of its two
arithmetics (GPU): remainders of frame and work tiles, boxes whose halos wrap
onto themselves, cells exactly one cutoff wide, lists that fill while the
candidates are tested, halos beyond the first, the second and every shared-
memory capacity. Two SER steps against the oracle, element by element, with
the tolerances of the parity tests (1e-11 in FP64, 2e-5 mixed: double and
float rounding of the pair arithmetic, accumulated over two steps)."""
import numpy as np
import pytest

from gpu_util import run_both

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "mixed": 2e-5}


def state(n, box, seed, float32, clump=None, cv=50.0):
    """Uniform positions; clump = (fraction, edge): that share of the particles in a corner cube."""
    rng = np.random.default_rng(seed)
    box = np.asarray(box, float)
    q = rng.random((n, 3)) * box
    if clump:
        m = int(clump[0] * n)
        q[:m] = rng.random((m, 3)) * clump[1]
    p = rng.standard_normal((n, 3))
    e = cv * (1 + 0.05 * rng.uniform(-1, 1, n))
    if float32:
        q = q.astype(np.float32).astype(np.float64)
        q = np.where(q >= box, 0.0, q)
        p = p.astype(np.float32).astype(np.float64)
    return q, p, e


CASES = {
    "wrapped": (90, (3.0, 3.2, 3.9), None),              # three cells: halos wrap onto themselves
    "exact_cells": (2592, (12.0, 8.0, 9.0), None),       # cells exactly r_cut wide
    "remainders": (6600, (13.4, 7.3, 19.9), None),       # 13 x 7 x 19 cells: frames of 6 and 1
    "full_lists": (2000, (4.6, 4.6, 4.6), None),         # ~86 neighbours: lists fill row by row
    "second_launch": (9000, (18.0, 9.0, 9.0), (0.25, 6.0)),    # a corner at 2.4x the mean density
    "beyond_shared": (27000, (30.0, 30.0, 30.0), (0.083, 8.0)),   # at 5.3x: the global path
}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", list(CASES))
def test_force_pass_edges(precision, case):
    n, box, clump = CASES[case]
    st = state(n, box, 7, precision == "mixed", clump)
    errs, _, _, _ = run_both([(n, box, 50.0, 1.0, (1, 1, 1))], precision, "SER", 2, dt=0.002, state=st)
    assert max(errs.values()) < TOL[precision], errs
