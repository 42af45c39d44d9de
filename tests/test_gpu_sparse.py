"""Sparse systems (GPU): whole frame tiles as work tiles, in one box and in
batches, boxes of four cells taken whole, remainders of one cell, a dense and
a sparse box in one handle. Two SER steps against the oracle, element by
element, with the tolerances of the parity tests (1e-11 in FP64, 2e-5 mixed:
double and float rounding of the pair arithmetic, accumulated over two
steps)."""
import pytest

from gpu_util import assert_parity

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
