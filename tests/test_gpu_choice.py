"""The automatic choice of sampler by the size of the call: few samples go to the kernels
that run a sample on a CTA (or with its state in shared memory), many samples of small
graphs and of graphs with long first walks, and calls in a workspace that holds the state
of few CTAs, to a lane per sample.  Each side was measured the faster one at these sizes
(by 1.4 or more); the counts of both are the oracle's in their own tests, and the sums of
the two are compared here."""
import numpy as np
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import (LAP_FORM_BLOCK, LAP_FORM_COMPACT, LAP_FORM_GROUP, LAP_FORM_SMALL, LAP_OPT_KERNEL,  # noqa: E402
                                        LAP_OPT_PATHS, LAP_STAT_LAST_FORM, LapGraph)

GRAPHS = {"ba": lambda n: I.ba(n, 5, seed=1), "er": lambda n: I.er(n, 10 / n, seed=1), "rmat": lambda n: I.rmat(13, 16, seed=1)}


@pytest.mark.parametrize("family,n,samples,ws,paths,form", [
    ("ba", 1000, 5000, 2 << 30, 0, LAP_FORM_BLOCK), ("ba", 1000, 200000, 2 << 30, 0, LAP_FORM_COMPACT),
    ("ba", 1000, 200000, 2 << 30, 1, LAP_FORM_COMPACT), ("ba", 4000, 1000, 8 << 30, 0, LAP_FORM_BLOCK),
    ("er", 1000, 10000, 2 << 30, 0, LAP_FORM_SMALL), ("er", 2000, 100000, 4 << 30, 0, LAP_FORM_COMPACT),
    ("er", 5000, 5000, 8 << 30, 0, LAP_FORM_BLOCK), ("er", 5000, 100000, 8 << 30, 0, LAP_FORM_COMPACT),
    ("er", 16000, 10000, 16 << 30, 0, LAP_FORM_BLOCK), ("er", 20000, 100000, 16 << 30, 0, LAP_FORM_COMPACT),
    ("er", 10000, 1000, 64 << 20, 0, LAP_FORM_BLOCK), ("er", 15000, 300, 30 << 20, 0, LAP_FORM_BLOCK),
    ("er", 40000, 5000, 400 << 20, 1, LAP_FORM_GROUP), ("er", 40000, 5000, 8 << 30, 1, LAP_FORM_BLOCK),
    ("rmat", 0, 40000, 16 << 30, 0, LAP_FORM_BLOCK),
    ("ba", 1400, 10000, 80 << 20, 1, LAP_FORM_COMPACT), ("ba", 500, 2000, 5 << 20, 0, LAP_FORM_COMPACT)])
def test_choice(family, n, samples, ws, paths, form):
    g = GRAPHS[family](n)
    out = []
    for kernel in (0, 2 if form in (LAP_FORM_BLOCK, LAP_FORM_SMALL) else 3):
        G = LapGraph(g.row_ptr, g.col, workspace_bytes=ws)
        try:
            G.set_option(LAP_OPT_PATHS, paths)
            G.set_option(LAP_OPT_KERNEL, kernel)
            G.set_root()
            G.sample(samples, 3)
            out.append(G.counts())
            if kernel == 0:
                assert G.stat(LAP_STAT_LAST_FORM) == form
        finally:
            G.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
