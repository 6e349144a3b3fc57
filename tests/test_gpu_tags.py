"""Calls of few and of many samples on one handle, with loop-included paths, on a graph
whose filter bits cover several nodes each (about 900,000 nodes on): the words of the
walks' departures and those of the Wilson runs share the workspace, and the border
between them moves with the number of samples in flight.  A word that an earlier call
has left must not be read as one of the present call: the counts are those of the
8-byte kernel for the same sample ids."""
import numpy as np
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import LAP_OPT_KERNEL, LAP_OPT_PATHS, LapGraph  # noqa: E402


def test_words_of_earlier_calls_are_not_read():
    g = I.ba(960000, 2, seed=1)
    sizes = [64] * 20 + [1400]
    out = []
    for kernel, calls in ((0, sizes), (1, [sum(sizes)])):
        G = LapGraph(g.row_ptr, g.col, workspace_bytes=16 << 30)
        try:
            G.set_option(LAP_OPT_PATHS, 1)
            G.set_option(LAP_OPT_KERNEL, kernel)
            G.set_root()
            for c in calls:
                G.sample(c, 7)
            out.append(G.counts())
        finally:
            G.close()
    for got, want in zip(*out):
        assert np.array_equal(got, want)
