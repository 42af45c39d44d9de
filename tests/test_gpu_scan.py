"""The cell scan beyond the tiles every block sums for itself (GPU): a sparse
box of 5.2 million cells, 2,500 scan tiles, against the oracle; and the same
particles in a box of one tile. Two SER steps, 1e-11 (double rounding of the
pair arithmetic)."""
import pytest

from gpu_util import assert_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,box", [(60000, (174.0, 173.0, 172.0)), (6000, (12.6, 12.7, 12.8)),
                                   (30000, (50.0, 50.0, 51.0))])
def test_scan_sizes(n, box):
    for _ in assert_parity([(n, box, 50.0, 1.0, (1, 1, 1))], "fp64", "SER", 2, 1e-11, (3,)):
        pass
