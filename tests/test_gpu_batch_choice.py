"""A batch's choice between branches and the persistent sampler, at sizes where one of them
was measured the faster one by 1.5 or more.  The counts of both are the same."""
import numpy as np
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import LAP_BOPT_LANES, LAP_BSTAT_BRANCHES, LapBatch  # noqa: E402


@pytest.mark.parametrize("graphs,samples,branches", [
    (lambda: [I.ba(500 + 5 * j, 3, seed=j) for j in range(300)], 64, False),
    (lambda: [I.ba(500 + 5 * j, 3, seed=j) for j in range(300)], 1000, False),
    (lambda: [I.er(1000, 0.01, seed=j) for j in range(64)], 4096, False),
    (lambda: [I.ba(20000, 5, seed=1), I.ba(30000, 4, seed=2)], 20000, True),
    (lambda: I.batch_graphs(I.batch_spec(24, 1000, 50000, seed0=0)), 256, True)],
    ids=["many_small_graphs", "small_graphs", "small_long_walks", "two_large", "uneven"])
def test_choice(graphs, samples, branches):
    gs = graphs()
    B = LapBatch([(g.row_ptr, g.col) for g in gs], workspace_bytes=4 << 30)
    try:
        B.run(samples, 5)
        B.sync()
        assert B.stat(LAP_BSTAT_BRANCHES) == (len(gs) if branches else 0)
        some = range(0, len(gs), max(1, len(gs) // 5))
        first = [B.counts(j) for j in some]
        B.set_option(LAP_BOPT_LANES, 20000)
        B.run(samples, 5)
        B.sync()
        assert B.stat(LAP_BSTAT_BRANCHES) == 0
        for j, a in zip(some, first):
            for x, y in zip(a, B.counts(j)):
                assert np.array_equal(x, y)
    finally:
        B.close()
