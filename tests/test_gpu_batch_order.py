"""LAP_BOPT_ORDER in a run on branches: with the smallest graphs first, most graphs are done
long before the batch is (their absorbed walks do not queue behind the longest ones), and
the smallest ones long before the largest."""
import numpy as np
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import LAP_BOPT_ORDER, LAP_BSTAT_BRANCHES, LapBatch  # noqa: E402


def test_smallest_first_completes_small_graphs_early():
    graphs = I.batch_graphs(I.batch_spec(60, 1000, 50000, seed0=3))
    n = np.array([g.n for g in graphs])
    B = LapBatch([(g.row_ptr, g.col) for g in graphs], workspace_bytes=4 << 30)
    try:
        B.set_option(LAP_BOPT_ORDER, 1)
        for _ in range(2):
            B.run(512, 5)
            B.sync()
        c = np.asarray(B.completion())
        assert B.stat(LAP_BSTAT_BRANCHES) == len(graphs)
    finally:
        B.close()
    small = n <= np.quantile(n, 0.25)
    assert c[small].min() < 0.1 * c.max()
    assert np.median(c) < 0.4 * c.max()
    assert np.median(c[small]) < np.median(c[~small])


def test_order_is_kept_where_both_samplers_would_run():
    """Enough samples of graphs with long first walks to fill the persistent sampler: graphs
    on branches would wait for it, so it takes them all when an order is asked for."""
    graphs = I.batch_graphs(I.batch_spec(60, 1000, 50000, seed0=3))
    B = LapBatch([(g.row_ptr, g.col) for g in graphs], workspace_bytes=16 << 30)
    try:
        branches, done = [], []
        for order in (0, 1):
            B.set_option(LAP_BOPT_ORDER, order)
            for _ in range(2):
                B.run(5000, 5)
                B.sync()
            branches.append(B.stat(LAP_BSTAT_BRANCHES))
            done.append(np.asarray(B.completion()))
    finally:
        B.close()
    assert 0 < branches[0] < len(graphs) and branches[1] == 0
    assert np.median(done[1]) < 0.4 * done[1].max()
