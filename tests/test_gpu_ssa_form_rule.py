"""Which form whole-replica SSA takes (GPU): the one expected to be faster for
the whole launch -- one replica or many, alike or uneven, more than the chip
holds at once, Lennard-Jones ones with long level tables -- and the same bits
from both."""
import numpy as np
import pytest

from gpu_util import make_state

pytestmark = pytest.mark.gpu

SOFT = dict(seed=9)
LJ = dict(seed=9, r_cut=2.5, sigma=2.0, potential=1, lj_eps=1.0, lj_r=1.0)


def handle(sizes, density, precision, prm):
    from paper_1507_06643_gb300 import dpde
    specs = [(n, ((n / density) ** (1 / 3),) * 3, 50.0, 1.0, (1, 1, 1)) for n in sizes]
    S = dpde.System(dpde.make_params(precision=precision, **prm),
                    [dpde.make_replica(n, box, cv, br) for n, box, cv, _, br in specs])
    return S, specs


def takes_levels(S):
    S.set_tuning(ssa_mode=0)
    classes = S.step_launches("SSA")
    S.set_tuning(ssa_mode=2)
    return S.step_launches("SSA") != classes


@pytest.mark.parametrize("sizes,density,precision,prm,levels", [
    # (us a step by levels / by classes)
    ([4000], 3.0, "mixed", SOFT, True),             # 431 / 838
    ([6000], 3.0, "mixed", SOFT, False),            # 474 / 294
    ([6000] * 64, 3.0, "mixed", SOFT, True),        # 597 / 901
    ([6000] * 152, 3.0, "mixed", SOFT, True),       # 813 / 1129
    ([6000] * 512, 3.0, "mixed", SOFT, False),      # 2982 / 2162
    ([500, 9900] * 16, 3.0, "mixed", SOFT, False),  # the large ones in the deferred launches
    ([6000], 3.0, "fp64", SOFT, False),             # 2576 / 1857
    ([7000] * 32, 3.0, "fp64", SOFT, True),         # 3518 / 8451
    ([500] * 1216, 0.8095, "mixed", LJ, True),      # 1583 / 4098 (phases), and 21612 without a schedule
    ([500, 2916, 500], 0.8095, "mixed", LJ, False),   # the second: ~77,000 entries, no schedule
])
def test_the_form_expected_to_be_faster(sizes, density, precision, prm, levels):
    S, _ = handle(sizes, density, precision, prm)
    assert takes_levels(S) == levels
    S.close()


@pytest.mark.parametrize("sizes,precision", [([6000] * 64, "mixed"), ([7000] * 8, "fp64"),
                                             ([3000, 900, 2600, 4900] * 16, "mixed")])
def test_both_forms_give_the_same_bits(sizes, precision):
    S, specs = handle(sizes, 3.0, precision, SOFT)
    assert takes_levels(S)
    st = make_state(specs, 5, precision == "mixed")
    out = []
    for mode in (2, 0):
        S.set_tuning(ssa_mode=mode)
        S.set_state(*st)
        S.step(2, 0.01, "SSA")
        out.append(S.get_state())
    S.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
