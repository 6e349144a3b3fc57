"""GPU parity of the small-graph kernel (sampler_small.cu), which automatic
calls take on graphs of up to 4096 nodes with long walks to the root (here, Barabasi-
Albert graphs rooted at a node of low degree): node counts around words of bits
and of draw bytes, the graph in shared or in global memory, samples around a
warp and a launch, loop-included paths, control-variate sums, and nodes drawn
more than 255 times.  Integers are bit-exact with the sequential oracle."""
import numpy as np
import pytest

import oracle
import oracle.cv as CV
from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import (LAP_OPT_PATHS, LAP_OPT_SLOTS, LAP_STAT_FALLBACKS,  # noqa: E402
                                        LAP_STAT_LAST_KERNEL, LapGraph)

CASES = [("two_nodes", lambda: I.path(2), 5, {}),
         ("n31", lambda: I.complete(31), 33, {}),
         ("n32", lambda: I.cycle(32), 65, {}),
         ("n33", lambda: I.ba(33, 2, seed=1), 1, dict(root=32)),
         ("n1000_many", lambda: I.ba(1000, 3, seed=2), 9000, dict(splits=[1, 8000, 999], root=999)),
         ("largest", lambda: I.ba(4096, 3, seed=3), 200, dict(trace=True, root=4095)),
         ("below_largest", lambda: I.ba(4095, 12, seed=4), 100, dict(root=4094)),
         ("dense_global_arcs", lambda: I.er(1500, 0.2, seed=5), 300, {}),
         ("slots", lambda: I.ba(700, 3, seed=6), 100, dict(slots=5, root=699)),
         ("paths", lambda: I.ba(900, 3, seed=7), 500, dict(paths=True, trace=True, root=899)),
         ("paths_one_lane", lambda: I.ba(900, 3, seed=7), 40, dict(paths=True, ws=1 << 20, slots=32, root=899)),
         ("drawn_often", lambda: I.path(200), 48, dict(root=0, trace=True)),
         ("drawn_often_paths", lambda: I.path(200), 48, dict(root=0, paths=True)),
         ("star", lambda: I.star(2000), 100, dict(root=7))]


@pytest.mark.parametrize("cv", [False, True], ids=["plain", "cv"])
@pytest.mark.parametrize("maker,omega,o", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_small_kernel_matches_oracle(maker, omega, o, cv):
    g = maker()
    paths = o.get("paths", False)
    phi = np.random.default_rng(3).uniform(0.0, 50.0, g.n)
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=o.get("ws", 1 << 26))
    try:
        if paths:
            G.set_option(LAP_OPT_PATHS, 1)
        if "slots" in o:
            G.set_option(LAP_OPT_SLOTS, o["slots"])
        v = G.set_root(o.get("root", -1))
        if cv:
            G.cv_set_potentials(torch.from_numpy(phi).cuda(), torch.from_numpy(phi).cuda())
        y = None
        if o.get("trace"):
            y = G.sample_trace(omega, 41)
        else:
            for part in o.get("splits", [omega]):
                G.sample(part, 41)
        c1, c2, s = G.counts()
        assert G.stat(LAP_STAT_LAST_KERNEL) == 3
        assert G.stat(LAP_STAT_FALLBACKS) == 0
        sums = G.cv_sums() if cv else None
    finally:
        G.close()
    if cv:
        h = CV.quantize_potential(phi)
        c, a1, a2, p2, _ = oracle.sample_cv(g.row_ptr, g.col, v, 41, 0, omega, h1=h, h2=h, paths=paths)
        for got, want in zip(sums, (a1, a2, p2)):
            assert np.array_equal(np.asarray(got), want)
    else:
        c = oracle.sample(g.row_ptr, g.col, v, 41, 0, omega, paths=paths)
    assert np.array_equal(c1, c.cnt1) and np.array_equal(c2, c.cnt2)
    if y is not None:
        assert all(np.array_equal(t.cpu().numpy().astype(np.uint64), w) for t, w in zip(y, (c.y1, c.y2)))
