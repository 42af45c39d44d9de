"""What the benchmark prints of its result: a line short enough for a reader
that keeps a few kilobytes of it, with every key, the shock's profile, which
only the report holds, and the form of the SSA that ran. CPU only."""
import json
import sys
from pathlib import Path

import numpy as np

sys.path.insert(0, str(Path(__file__).resolve().parents[1]))

import bench  # noqa: E402


def profile():
    rng = np.random.default_rng(1)
    z = rng.random(400000) * 800.0
    z[0] = 800.0                       # the far end belongs to the last slab
    return bench.eps_profile([(k, z, 100.0 + z / 16.0) for k in ("t0", "half", "end")], 800.0, [0.0, 50.0, 100.0],
                             bench.SHOCK_SLABS)


def test_profile_holds_the_slab_means():
    prof = profile()
    mid = (np.arange(800) + 0.5) * prof["slab_width"]
    for k in ("t0", "half", "end"):
        # all particles of a slab lie within half its width: 0.5 / 16
        assert np.max(np.abs(np.asarray(prof[k]) - (100.0 + mid / 16.0))) < 0.032
    assert bench.slab_means(np.array([0.1]), np.array([7.0]), 1.0, 4).tolist() == [7.0, 0.0, 0.0, 0.0]


def test_line_is_short_and_keeps_its_keys():
    phase = {"bound": "alu", "kernel": "k", "phase": "ssa", "achieved": 1 / 3, "peak": 2 / 3, "unit": "Gop/s",
             "frac": 1 / 3, "traffic": None, "peak_source": "p" * 60}
    out = {"metric": "m", "value": 1e9 / 3, "ms_per_step": 2 / 3, "config": {"tuning": {"block": 256}, "dt": 0.01},
           "roofline": phase, "roofline_phases": {str(k): phase for k in range(5)},
           "shock": {"value": 1e9 / 3, "eps_profile": profile(), "tuning": {}}, "parity": {"fp64": 1e-13 / 3, "sample": "s"},
           "clocks": None}
    assert len(json.dumps(out)) > 20000
    line = bench.line_of(out)
    assert len(json.dumps(line)) < 1500
    assert line.keys() == out.keys()
    assert line["value"] == out["value"] and line["config"] == out["config"]
    assert line["shock"] == {"value": 333333000.0} and line["parity"] == {"fp64": 3.33333e-14}
    assert line["roofline_phases"]["0"] == {"kernel": "k", "frac": 0.333333}


class Launches:
    """A handle whose level form is possible or not."""

    def __init__(self, levels):
        self.levels, self.mode = levels, 2

    def set_tuning(self, ssa_mode):
        self.mode = ssa_mode

    def step_launches(self, scheme):
        return 16 if self.mode == 2 and self.levels else 35


def test_the_form_that_runs():
    for levels, form in ((True, 2), (False, 0)):
        S = Launches(levels)
        assert bench.ssa_form(S, "SSA", 2) == form and S.mode == 2
    assert bench.ssa_form(Launches(True), "SSA", 1) == 0
    assert bench.ssa_form(Launches(True), "HYBRID", 1) == 1
    assert bench.ssa_form(Launches(False), "SER", 2) == 2
