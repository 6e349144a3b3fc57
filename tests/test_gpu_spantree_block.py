"""SpanTree sums of the block kernel's trees against those of the 8-byte
Wilson kernel (LAP_OPT_KERNEL = 1): the same trees, so the same integers, for
every size and workspace, and between ordinary samples."""
import numpy as np
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import LAP_OPT_KERNEL, LAP_OPT_SLOTS, LapGraph  # noqa: E402


@pytest.mark.parametrize("maker,splits,root", [(lambda: I.path(2), [5], 0), (lambda: I.ba(33, 2, seed=1), [64], -1),
                                               (lambda: I.ba(4097, 3, seed=2), [1, 200], -1),
                                               (lambda: I.rmat(14, 8, seed=3), [100], 77), (lambda: I.path(300), [20], 299),
                                               (lambda: I.er(12000, 6 / 12000, seed=4), [150], -1)],
                         ids=["two_nodes", "n33", "n4097", "rmat", "path", "parts"])
def test_trees_equal_wide_kernel(maker, splits, root):
    g = maker()
    out = []
    for kernel, ws, slots in ((1, 1 << 28, 0), (0, 1 << 28, 0), (0, 1 << 28, 3), (0, 8 * g.n * 300, 0)):
        G = LapGraph(g.row_ptr, g.col, workspace_bytes=max(ws, 8192))
        try:
            G.set_option(LAP_OPT_KERNEL, kernel)
            if slots:
                G.set_option(LAP_OPT_SLOTS, slots)
            G.set_root(root)
            for c in splits:
                G.sample(10, 5)
                G.spantree_sample(c, 9)
            c1, c2, s = G.counts()
            out.append([np.asarray(x) for x in G.spantree_sums()[:3]] + [c1, c2])
        finally:
            G.close()
    for o in out[1:]:
        for x, y in zip(out[0], o):
            assert np.array_equal(x, y)
