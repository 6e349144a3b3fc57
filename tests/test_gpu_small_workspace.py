"""The small-graph kernel in workspaces that do not hold all samples of a call: fewer
samples in flight, down to one, with a share for the loop-included paths' words.  The
sizes lie around one sample's state and around a warp's and a launch's samples; integers
are bit-exact with the sequential oracle."""
import numpy as np
import pytest

import oracle
from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import LAP_FORM_SMALL, LAP_OPT_PATHS, LAP_OPT_SLOTS, LAP_STAT_LAST_FORM, LapGraph  # noqa: E402


@pytest.mark.parametrize("paths", [0, 1], ids=["own_draws", "paths"])
@pytest.mark.parametrize("n,units,samples,slots", [(300, 64, 256, 0), (1000, 2, 30, 0), (1000, 3, 30, 0), (999, 40, 200, 0),
                                                   (1000, 700, 3000, 0), (700, 60, 100, 7), (2000, 160, 500, 0)])
def test_tight_workspaces(n, units, samples, slots, paths):
    g = I.er(n, 10 / n, seed=2)
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=units * 8 * g.n)
    try:
        G.set_option(LAP_OPT_PATHS, paths)
        G.set_option(LAP_OPT_SLOTS, slots)
        v = G.set_root()
        G.sample(samples, 17)
        c1, c2, s = G.counts()
        # One sample: its stack and words (6 n), with paths one walk's words and 3/8 of another's.
        if units * 8 * g.n >= 600 + (17 if paths else 6) * g.n:
            assert G.stat(LAP_STAT_LAST_FORM) == LAP_FORM_SMALL
    finally:
        G.close()
    c = oracle.sample(g.row_ptr, g.col, v, 17, 0, samples, paths=bool(paths))
    assert np.array_equal(c1, c.cnt1) and np.array_equal(c2, c.cnt2)
    assert int(s[1]) == c.sum_y1 and int(s[2]) == c.sum_y2
