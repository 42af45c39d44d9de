"""Sparse systems (GPU): whole frame tiles as work tiles, in one box and in
batches, boxes of four cells taken whole, remainders of one cell, a dense and
a sparse box in one handle. Two SER steps against the oracle, element by
element, with the tolerances of the parity tests (1e-11 in FP64, 2e-5 mixed:
double and float rounding of the pair arithmetic, accumulated over two
steps)."""
import numpy as np
import pytest

from gpu_util import assert_parity, run_both

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "mixed": 2e-5}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("boxes", [
    [(1500, (25.0, 13.3, 19.9))],                    # 0.23 a cell unit: frames of 6 and of 1
    [(300, (10.0, 10.0, 10.0))] * 12,                # 0.3
    [(190, (4.05, 4.0, 4.9))] * 9,                   # four cells an axis, dense
    [(40, (9.0, 9.0, 9.0)), (600, (7.0, 7.0, 7.0)), (0, (8.0, 8.0, 8.0)), (5, (16.0, 3.0, 5.0))],
])
def test_sparse_boxes(boxes, precision):
    specs = [(n, box, 50.0, 1.0, (1, 1, 1)) for n, box in boxes]
    for _ in assert_parity(specs, precision, "SER", 2, TOL[precision], (3,), dt=0.002):
        pass


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("bricks,walls", [((1, 1, 1), (0, 0.0)), ((7, 5, 4), (0, 0.0)), ((1, 1, 1), (1, -0.5))])
def test_observables_of_a_very_sparse_box(bricks, walls, precision):
    """950,000 cells for 3,000 particles, half of them in a drop across the
    periodic corner: the pair sums particle by particle, rows of cells that
    are neighbours in memory and rows that a domain or the box cuts, against
    the oracle (the parity tolerance, on sums: relative to the sum)."""
    box = (101.0, 97.5, 99.2)
    rng = np.random.default_rng(11)
    n = 3000
    q = rng.random((n, 3)) * np.asarray(box)
    q[:n // 2] = (rng.random((n // 2, 3)) - 0.5) * 8.0
    if walls[0]:
        q[:n // 2, 2] += 4.0
    q = np.mod(q, np.asarray(box))
    p = rng.standard_normal((n, 3))
    if precision == "mixed":
        q = q.astype(np.float32).astype(np.float64)
        p = p.astype(np.float32).astype(np.float64)
        q = np.where(q >= np.asarray(box), 0.0, q)
    e = 50.0 * (1 + 0.05 * rng.uniform(-1, 1, n))
    errs, _, (_, _, _, obs), ref = run_both([(n, box, 50.0, 1.0, bricks)], precision, "SER", 1, dt=0.002,
                                            state=(q, p, e), walls=walls)
    assert max(errs.values()) < TOL[precision], errs
    o = ref.observables(0)
    assert o["U"] > 100.0
    for k in ("U", "Tpot_num", "Tpot_den"):
        assert abs(obs[0][k] - o[k]) <= 10 * TOL[precision] * abs(o[k]), (k, obs[0][k], o[k])


@pytest.mark.parametrize("precision,scheme", [("fp64", "SER"), ("mixed", "SER"), ("fp64", "HYBRID")])
@pytest.mark.parametrize("n,box", [(6000, (28.0, 25.2, 31.0)), (1000, (61.0, 60.0, 59.0))])
def test_a_drop_in_a_thin_gas(n, box, precision, scheme):
    """780 particles at 3.6 a cell unit in the corner of a gas of 0.24 or
    0.001: the first launch defers the drop's work tiles, whose halos hold
    many times the mean."""
    rng = np.random.default_rng(12)
    q = rng.random((n, 3)) * np.asarray(box)
    q[:780] = rng.random((780, 3)) * 6.0
    p = rng.standard_normal((n, 3))
    if precision == "mixed":
        q = q.astype(np.float32).astype(np.float64)
        p = p.astype(np.float32).astype(np.float64)
    e = 50.0 * (1 + 0.05 * rng.uniform(-1, 1, n))
    errs, _, _, _ = run_both([(n, box, 50.0, 1.0, (2, 1, 3))], precision, scheme, 2, dt=0.002, state=(q, p, e))
    assert max(errs.values()) < TOL[precision], errs


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_clump_beyond_every_capacity(precision):
    """A fluid at 3 a cell unit (work tiles of 6 x 6 x 2 cells) with 8 x 8 x 4
    cells at 9.5: ~2,430 particles in the halo of the tile inside, more than
    the ~2,070 of the second launch, so that tile goes through global memory,
    several threads a cell."""
    box = (42.2, 42.2, 42.2)
    n, extra = 222000, 1664
    rng = np.random.default_rng(13)
    q = rng.random((n + extra, 3)) * np.asarray(box)
    cell = box[0] / 42
    q[:extra] = np.array([5.0, 5.0, 5.0]) * cell + rng.random((extra, 3)) * np.array([8.0, 8.0, 4.0]) * cell
    p = rng.standard_normal((n + extra, 3))
    if precision == "mixed":
        q = q.astype(np.float32).astype(np.float64)
        q = np.where(q >= np.asarray(box), 0.0, q)
        p = p.astype(np.float32).astype(np.float64)
    e = 50.0 * (1 + 0.05 * rng.uniform(-1, 1, n + extra))
    errs, _, _, _ = run_both([(n + extra, box, 50.0, 1.0, (1, 1, 1))], precision, "SER", 1, dt=0.002, state=(q, p, e))
    assert max(errs.values()) < TOL[precision], errs
