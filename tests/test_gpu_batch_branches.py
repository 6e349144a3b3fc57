"""GPU parity of batch runs on branches (a graph's samples by the kernels of
single graphs, graphs side by side): more graphs than branches, sizes around
the kernels' ranges, a shared CSR with two roots, path starts changed between
runs, loop-included paths, a workspace that holds one branch or none, and the
change to the persistent sampler by a launch option.  Integers are bit-exact
with the sequential oracle."""
import numpy as np
import pytest

import oracle
from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import (LAP_BOPT_LANES, LAP_BOPT_ORDER, LAP_BOPT_PATHS, LAP_BSTAT_GRAPH_CAPTURES,  # noqa: E402
                                        LapBatch)


def graphs20():
    g = [I.path(2), I.star(33), I.path(200), I.ba(1000, 3, seed=1), I.ba(4096, 3, seed=2), I.ba(4097, 3, seed=3),
         I.rmat(13, 8, seed=4), I.ba(20000, 4, seed=5), I.er(3000, 0.003, seed=6)]
    return g + [I.ba(300 + 37 * j, 2, seed=j) for j in range(11)]


def check(B, graphs, seed, k, paths=False, starts=None):
    for j, g in enumerate(graphs):
        v = int(B.roots[j])
        c = oracle.sample(g.row_ptr, g.col, v, seed, 0, k, keep_per_sample=False, paths=paths,
                          path_start=-1 if starts is None else starts[j])
        c1, c2, sums = B.counts(j)
        assert np.array_equal(c1, c.cnt1) and np.array_equal(c2, c.cnt2), j
        assert int(sums[1]) == c.sum_y1 and int(sums[2]) == c.sum_y2, j


@pytest.mark.parametrize("paths", [False, True], ids=["own_draws", "paths"])
@pytest.mark.parametrize("order,ws", [(0, 1 << 30), (1, 1 << 26), (2, 6 << 20), (0, 1 << 19)],
                         ids=["branches", "smaller_shares", "few_branches", "persistent"])
def test_branches_match_oracle(order, ws, paths):
    graphs = graphs20()
    shared = graphs[3]
    B = LapBatch([(g.row_ptr, g.col) for g in graphs + [shared]], roots=[-1] * len(graphs) + [17], workspace_bytes=ws)
    try:
        B.set_option(LAP_BOPT_ORDER, order)
        if paths:
            B.set_option(LAP_BOPT_PATHS, 1)
        for seed in (11, 12):
            B.run(24, seed)
            check(B, graphs + [shared], seed, 24, paths)
            assert np.all(np.asarray(B.completion()) > 0.0)
    finally:
        B.close()


def test_path_starts_and_options_between_runs():
    graphs = graphs20()[3:8]
    B = LapBatch([(g.row_ptr, g.col) for g in graphs], workspace_bytes=1 << 28)
    try:
        B.run(16, 3)
        check(B, graphs, 3, 16)
        starts = [5, -1, 0, 77, 4000]
        for j, s in enumerate(starts):
            B.set_path_start(j, s)
        B.run(16, 3)
        check(B, graphs, 3, 16, starts=starts)
        assert B.stat(LAP_BSTAT_GRAPH_CAPTURES) == 1       # starts are read at run time
        B.set_option(LAP_BOPT_LANES, 40)
        B.run(16, 3)
        check(B, graphs, 3, 16, starts=starts)
        B.set_option(LAP_BOPT_LANES, 0)
        B.run(16, 3)
        check(B, graphs, 3, 16, starts=starts)
        assert B.stat(LAP_BSTAT_GRAPH_CAPTURES) == 3
    finally:
        B.close()
