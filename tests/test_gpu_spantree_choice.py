"""SpanTree's choice of sampler: the block kernel for few trees and for large graphs, a lane
per tree for many trees of small graphs (measured the faster one at these sizes by 2 or
more).  The sums of both samplers are the same integers, also where one call changes from
one to the other (its last launch has few trees)."""
import numpy as np
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import (LAP_FORM_BLOCK, LAP_FORM_WIDE, LAP_OPT_KERNEL, LAP_STAT_TREE_FORM,  # noqa: E402
                                        LapGraph)


def er(n):
    return I.er(n, 10 / n, seed=1)


@pytest.mark.parametrize("g,trees,lanes,form", [
    (er(1000), 512, 32768, LAP_FORM_BLOCK), (er(1000), 32768, 32768, LAP_FORM_WIDE),
    (I.ba(300, 3, seed=1), 20000, 32768, LAP_FORM_WIDE), (I.ba(1000, 5, seed=1), 32768, 32768, LAP_FORM_WIDE),
    (er(4000), 20000, 32768, LAP_FORM_WIDE), (I.ba(10000, 5, seed=1), 4096, 32768, LAP_FORM_BLOCK),
    (er(10000), 1000, 32768, LAP_FORM_BLOCK), (er(10000), 32768, 32768, LAP_FORM_WIDE), (er(1000), 8200, 2048, None)],
    ids=["er_few", "er_many", "n300", "ba_many", "er_4000", "ba_10k", "er_10k", "er_10k_many", "changes"])
def test_trees_by_size(g, trees, lanes, form):
    out = []
    for kernel in (0, 3 if form == LAP_FORM_WIDE else 1):
        G = LapGraph(g.row_ptr, g.col, workspace_bytes=8 * g.n * lanes)
        try:
            G.set_option(LAP_OPT_KERNEL, kernel)
            G.set_root()
            G.spantree_sample(trees, 9)
            if kernel == 0 and form:
                assert G.stat(LAP_STAT_TREE_FORM) == form
            out.append([np.asarray(x) for x in G.spantree_sums()[:3]])
        finally:
            G.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
