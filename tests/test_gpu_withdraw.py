"""Withdrawn samples of the one-CTA-per-sample kernel (a sample without progress gives back
what it has counted, and is run again with the 8-byte kernel): LAP_OPT_WITHDRAW makes
samples withdraw at their start (the early phase's counts alone), before the sweeps and at
their end.  Counts, traces, control-variate sums, batches and SpanTree sums are those of
the sequential oracle, or of a run without withdrawals."""
import numpy as np
import pytest

import oracle
import oracle.cv as CV
from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import (LAP_BOPT_WITHDRAW, LAP_BSTAT_BRANCHES, LAP_BSTAT_RERUNS, LAP_FORM_BLOCK,  # noqa: E402
                                        LAP_FORM_WIDE, LAP_OPT_PATHS, LAP_OPT_WITHDRAW, LAP_STAT_FALLBACKS,
                                        LAP_STAT_LAST_FORM, LAP_STAT_TREE_FORM, LapBatch, LapGraph)

GRAPHS = {"ba": lambda: I.ba(5001, 3, seed=1), "hubs": lambda: I.rmat(14, 8, seed=8),
          "long_walks": lambda: I.er(12000, 6 / 12000, seed=9)}


@pytest.mark.parametrize("every", [1, 5])
@pytest.mark.parametrize("paths", [False, True], ids=["own_draws", "paths"])
@pytest.mark.parametrize("cv", [False, True], ids=["plain", "cv"])
@pytest.mark.parametrize("name", list(GRAPHS))
def test_counts_and_traces(name, cv, paths, every):
    g = GRAPHS[name]()
    calls = [30, 17]
    phi = np.random.default_rng(3).uniform(0.0, 50.0, g.n)
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=1 << 28)
    try:
        G.set_option(LAP_OPT_PATHS, int(paths))
        G.set_option(LAP_OPT_WITHDRAW, every)
        v = G.set_root()
        if cv:
            G.cv_set_potentials(torch.from_numpy(phi).cuda(), torch.from_numpy(phi).cuda())
        y = []
        for c in calls:
            t = (G.sample_trace_cv if cv else G.sample_trace)(c, 41)
            G.sync()
            y.append([x.cpu().numpy() for x in t])
            assert G.stat(LAP_STAT_LAST_FORM) == LAP_FORM_BLOCK
        assert G.stat(LAP_STAT_FALLBACKS) == sum((c + every - 1) // every for c in calls)
        c1, c2, s = G.counts()
        sums = G.cv_sums() if cv else None
    finally:
        G.close()
    n = sum(calls)
    if cv:
        h = CV.quantize_potential(phi)
        c, a1, a2, p2, m2 = oracle.sample_cv(g.row_ptr, g.col, v, 41, 0, n, h1=h, h2=h, paths=paths)
        for got, want in zip(sums, (a1, a2, p2)):
            assert np.array_equal(np.asarray(got), want)
    else:
        c = oracle.sample(g.row_ptr, g.col, v, 41, 0, n, paths=paths)
    assert np.array_equal(c1, c.cnt1) and np.array_equal(c2, c.cnt2)
    assert int(s[1]) == c.sum_y1 and int(s[2]) == c.sum_y2
    for j, want in enumerate((c.y1, c.y2)):
        assert np.array_equal(np.concatenate([t[j] for t in y]).astype(np.uint64), want)


def test_batch():
    graphs = [I.ba(5001, 3, seed=1), I.ba(300, 2, seed=2), I.rmat(12, 8, seed=3), I.ba(6000, 4, seed=4)]
    B = LapBatch([(g.row_ptr, g.col) for g in graphs], workspace_bytes=1 << 28)
    try:
        for every, rerun in ((0, False), (4, True), (1, True), (0, False)):
            B.set_option(LAP_BOPT_WITHDRAW, every)
            B.run(21, 9)
            B.sync()
            assert B.stat(LAP_BSTAT_BRANCHES) == len(graphs)
            assert (B.stat(LAP_BSTAT_RERUNS) > 0) == rerun
            for j, g in enumerate(graphs):
                c = oracle.sample(g.row_ptr, g.col, int(B.roots[j]), 9, 0, 21, keep_per_sample=False)
                c1, c2, sums = B.counts(j)
                assert np.array_equal(c1, c.cnt1) and np.array_equal(c2, c.cnt2), (every, j)
                assert int(sums[1]) == c.sum_y1 and int(sums[2]) == c.sum_y2, (every, j)
    finally:
        B.close()


def test_spantree():
    g = I.ba(5001, 3, seed=1)
    out = []
    for every in (0, 7):
        G = LapGraph(g.row_ptr, g.col, workspace_bytes=1 << 28)
        try:
            G.set_option(LAP_OPT_WITHDRAW, every)
            G.set_root()
            G.sample(10, 5)
            G.spantree_sample(40, 9)
            assert G.stat(LAP_STAT_TREE_FORM) == (LAP_FORM_WIDE if every else LAP_FORM_BLOCK)
            G.sample(10, 5)
            out.append([np.asarray(x) for x in G.spantree_sums()[:3]] + list(G.counts()))
        finally:
            G.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
