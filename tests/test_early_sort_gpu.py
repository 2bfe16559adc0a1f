"""Early sorts of a small species (needs a GB300): a beam whose particles all
reach the end of the tiles' drift allowance in the same step.

The beam moves 0.64 cells per step along x and is sorted at step 0 only, so
no particle escapes in the first two pushes and about 2.6 % do in the third
(a tile is 16 cells wide and lends one cell).  Whenever a push sends more than
0.5 % of the species (and 1024 particles) down the escape path, the species is
sorted at the next step.
"""
import numpy as np
import pytest

from paper_1503_02464_gb300 import synth
from paper_1503_02464_gb300.sim import Simulation

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_sorted_at_the_step_after_the_escapes(precision):
    wl = synth.small(2, (256, 64), 2, 8, 0.0, 19)
    p = wl.particles(0)
    n = len(p["x"])
    p["ux"] = np.full(n, 3.0)
    p["w"] = np.full(n, 1e-9)  # a test beam: its fields do nothing
    move = wl.dt / wl.d[0] * 3.0 / np.sqrt(10.0)
    assert 0.6 < move < 0.66
    s = Simulation.from_workload(wl, precision=precision, sort_every=1000)
    k = s.add_species(-1.0, 1.0, n)
    s.load(k, p)
    limit = max(n // 200, 1024)
    due, early, escaped = False, 0, 0
    seen = []
    for step in range(12):
        s.step(1)
        s.sync()  # the push's count is there before the next step is enqueued
        d = s.diag()
        seen.append((d["n_escaped"] - escaped, d["n_sorts_adaptive"] - early))
        assert seen[-1][1] == (1 if due else 0), seen
        due = seen[-1][0] > limit
        early, escaped = d["n_sorts_adaptive"], d["n_escaped"]
    assert early >= 2, seen
    s.close()
