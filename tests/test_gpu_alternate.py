"""Calls of different sizes on one handle, so that samplers with different layouts of the
workspace take turns, SpanTree among them: the counts are those of the 8-byte kernel for
the same sample ids."""
import numpy as np
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import (LAP_FORM_BLOCK, LAP_FORM_COMPACT, LAP_FORM_SMALL, LAP_OPT_KERNEL,  # noqa: E402
                                        LAP_OPT_PATHS, LAP_STAT_LAST_FORM, LapGraph)


@pytest.mark.parametrize("paths", [0, 1], ids=["own_draws", "paths"])
@pytest.mark.parametrize("g,few", [(I.ba(1000, 5, seed=1), LAP_FORM_BLOCK), (I.er(1000, 0.01, seed=1), LAP_FORM_SMALL)],
                         ids=["block", "small"])
def test_samplers_take_turns(g, few, paths):
    sizes = [100, 200000, 70, 1000, 0, 200000, 0, 300, 17]          # 0: trees between the calls
    out = []
    for kernel in (0, 1):
        G = LapGraph(g.row_ptr, g.col, workspace_bytes=2 << 30)
        try:
            G.set_option(LAP_OPT_PATHS, paths)
            G.set_option(LAP_OPT_KERNEL, kernel)
            G.set_root()
            for c in sizes if kernel == 0 else [sum(sizes)]:
                if c == 0:
                    G.spantree_sample(40, 9)
                    continue
                G.sample(c, 7)
                if kernel == 0:
                    assert G.stat(LAP_STAT_LAST_FORM) == (LAP_FORM_COMPACT if c > 10000 else few)
            if kernel:
                for _ in range(sizes.count(0)):
                    G.spantree_sample(40, 9)
            out.append(list(G.counts()) + [np.asarray(x) for x in G.spantree_sums()[:3]])
        finally:
            G.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
