"""The SER sweeps and the SEM sweep at the edges of their flat lists (GPU): warps with one entry,
a last warp of one particle, lists that end on and straddle a window of the
shared-memory list, particles without cross-domain pairs between ones that
have them. Two steps against the oracle, element by element, with the
tolerances of the parity tests (1e-11 in FP64, 2e-5 mixed: double and float
rounding of the pair arithmetic, accumulated over two steps)."""
import pytest

from gpu_util import assert_parity

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "mixed": 2e-5}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,edge,bricks,scheme", [
    (2, 3.0, (1, 1, 1), "SER"), (33, 3.0, (1, 1, 1), "SER"),
    (161, 3.0, (1, 1, 1), "SER"),       # ~25 neighbours: ~800 entries a warp, two or four windows
    (700, 3.6, (1, 1, 1), "SER"),       # ~63 neighbours, ~2000 entries
    (33, 3.0, (1, 1, 1), "SEM"), (700, 3.6, (1, 1, 1), "SEM"),
    (1500, 7.3, (2, 2, 1), "HYBRID"),   # cross pairs only along the domain faces
])
def test_sweeps_edges(n, edge, bricks, scheme, precision):
    specs = [(n, (edge,) * 3, 50.0, 1.0, bricks)]
    for _ in assert_parity(specs, precision, scheme, 2, TOL[precision], (3, 4, 5), dt=0.002):
        pass
