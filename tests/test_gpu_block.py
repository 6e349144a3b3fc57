"""GPU parity of the one-CTA-per-sample kernel (sampler_block.cu), which
automatic calls take on graphs above the small-graph kernel's range, at the
sizes where it can go wrong: node counts around a word of tree bits, samples
around the number in flight, a workspace too small for the early phase or for
more than one sample, long first walks whose tables fit a part of the call only,
loop-included paths, control-variate sums, and cycles
longer than the bookkeeping's short forms.  Integers are bit-exact with the
sequential oracle."""
import numpy as np
import pytest

import oracle
from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import oracle.cv as CV  # noqa: E402
from paper_2311_10290_gb300.lap import (LAP_OPT_PATHS, LAP_OPT_SLOTS, LAP_STAT_FALLBACKS, LAP_STAT_LAST_KERNEL,  # noqa: E402
                                        LapGraph)


def grid(k):
    """k x k grid: long walks and cycles of many lengths."""
    x = np.arange(k * k).reshape(k, k)
    e = np.concatenate([np.stack([x[:, :-1].ravel(), x[:, 1:].ravel()], 1), np.stack([x[:-1].ravel(), x[1:].ravel()], 1)])
    return I.from_edges(k * k, e)


def crossed_pairs():
    """A star with its leaves paired 8192 ids apart but for the lowest bit: the locks
    (13 low id bits) of neighbouring pairs coincide crosswise."""
    i, leaf = np.arange(2, 8192), np.arange(1, 16384)
    return I.from_edges(16384, np.concatenate([np.stack([i, 8192 + (i ^ 1)], 1), np.stack([0 * leaf, leaf], 1)]))


CASES = [("word_minus_1", lambda: I.ba(4127, 3, seed=1), 40, {}),
         ("word", lambda: I.ba(4128, 2, seed=2), 1, {}),
         ("word_plus_1", lambda: I.ba(4129, 4, seed=3), 33, dict(trace=True)),
         ("many_samples", lambda: I.ba(4500, 3, seed=4), 3000, dict(splits=[1, 2499, 500])),
         ("slots", lambda: I.ba(30000, 3, seed=5), 64, dict(slots=7)),
         ("no_early_tables", lambda: I.ba(30000, 3, seed=5), 12, dict(ws=1870000)),
         ("one_in_flight", lambda: I.ba(30000, 3, seed=6), 12, dict(ws=3 << 20)),
         ("paths", lambda: I.ba(6000, 3, seed=7), 100, dict(paths=True, trace=True)),
         ("hubs", lambda: I.rmat(14, 8, seed=8), 64, dict(trace=True)),
         ("star", lambda: I.star(5000), 64, dict(root=17)),
         ("grid", lambda: grid(66), 24, dict(root=0)),
         ("parts", lambda: I.er(12000, 6 / 12000, seed=9), 300, dict(ws=24 << 20, trace=True)),
         ("long_paths", lambda: I.er(70000, 4 / 70000, seed=10), 8, {}),
         ("crossed_pairs", crossed_pairs, 200, dict(no_reruns=True))]


@pytest.mark.parametrize("cv", [False, True], ids=["plain", "cv"])
@pytest.mark.parametrize("maker,omega,o", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_block_kernel_matches_oracle(maker, omega, o, cv):
    g = maker()
    paths = o.get("paths", False)
    rng = np.random.default_rng(3)
    phi = rng.uniform(0.0, 50.0, g.n)
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=o.get("ws", 1 << 28))
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
            y = [t.cpu().numpy().astype(np.uint64) for t in G.sample_trace(omega, 41)]
        else:
            for part in o.get("splits", [omega]):
                G.sample(part, 41)
        c1, c2, s = G.counts()
        assert G.stat(LAP_STAT_LAST_KERNEL) == 3
        assert not o.get("no_reruns") or G.stat(LAP_STAT_FALLBACKS) == 0
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
        assert np.array_equal(y[0], c.y1) and np.array_equal(y[1], c.y2)
