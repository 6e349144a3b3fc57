"""GPU row sums (rows.cuh) at the degrees where a row changes hands: one
thread, one warp, one CTA.  A breadth-first search, the FP64 solve and the
features all run on them."""
import numpy as np
import pytest

import oracle.cg as CG
import oracle.cv as CV
from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import LapGraph  # noqa: E402


def hub_graph(degrees, n=3000):
    """A cycle with chords from node j * 100 that give it degrees[j] (and one more for
    each earlier hub whose chords reach it)."""
    e = [(i, (i + 1) % n) for i in range(n)]
    for j, d in enumerate(degrees):
        h = j * 100
        e += [(h, (h + 2 + k) % n) for k in range(d - 2)]
    return I.from_edges(n, np.array(e))


@pytest.mark.parametrize("degrees,n", [((47, 48, 49, 50), 3000), ((255, 255, 255, 255), 3000),
                                       ((1024, 2990, 600, 700, 800), 3000), ((33,), 255), ((2,), 257)],
                         ids=["thread_warp", "warp_cta", "hubs", "one_block", "cycle"])
def test_rows_match_oracle(degrees, n):
    g = hub_graph(degrees, n)
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=1 << 24)
    try:
        for root in (-1, n - 1):
            v = G.set_root(root)
            f = G.features().cpu().numpy().astype(np.float64)
            np.testing.assert_allclose(f, CV.features(g.row_ptr, g.col, v).astype(np.float32), rtol=2e-6, atol=1e-6)
            b = np.random.default_rng(1).standard_normal(n)
            x, it, res = G.lv_solve(b)
            y, it2, _ = G.lv_solve(b)
            want, _, _ = CG.solve_lv(g.row_ptr, g.col, v, b)
            assert res <= 1e-12 and it > 0 and it2 == it and np.array_equal(x, y)
            np.testing.assert_allclose(x, want, rtol=1e-9, atol=1e-9 * np.abs(want).max())
    finally:
        G.close()
