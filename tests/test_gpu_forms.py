"""Which sampler a call takes.  The parity tests of the block kernel, of the small-graph
kernel, of SpanTree trees and of batches on branches compare counts alone, which every
sampler has in common; here their calls are made again and the sampler is looked at."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import test_gpu_block as block  # noqa: E402
import test_gpu_small as small  # noqa: E402
from test_gpu_batch_branches import graphs20  # noqa: E402
from paper_2311_10290_gb300 import inputs as I  # noqa: E402
from paper_2311_10290_gb300.lap import (LAP_BOPT_LANES, LAP_BSTAT_BRANCHES, LAP_FORM_BLOCK, LAP_FORM_COMPACT,  # noqa: E402
                                        LAP_FORM_GROUP, LAP_FORM_SMALL, LAP_FORM_WIDE, LAP_OPT_KERNEL, LAP_OPT_PATHS,
                                        LAP_OPT_SLOTS, LAP_OPT_WALKERS, LAP_STAT_LAST_FORM, LAP_STAT_TREE_FORM,
                                        LapBatch, LapGraph)


def form_of(g, calls, workspace, options=(), root=-1):
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=workspace)
    try:
        for o, v in options:
            G.set_option(o, v)
        G.set_root(root)
        forms = []
        for c in calls:
            G.sample(c, 41)
            forms.append(G.stat(LAP_STAT_LAST_FORM))
        return forms
    finally:
        G.close()


@pytest.mark.parametrize("module,form,default_ws", [(block, LAP_FORM_BLOCK, 1 << 28), (small, LAP_FORM_SMALL, 1 << 26)],
                         ids=["block", "small"])
def test_parity_cases_take_their_kernel(module, form, default_ws):
    for name, maker, omega, o in module.CASES:
        if name == "no_early_tables":
            continue            # LapGraph lends whole multiples of 8 n bytes: not enough for the block kernel
        options = [(LAP_OPT_PATHS, 1)] * o.get("paths", False) + ([(LAP_OPT_SLOTS, o["slots"])] if "slots" in o else [])
        calls = o.get("splits", [omega])
        assert form_of(maker(), calls, o.get("ws", default_ws), options, o.get("root", -1)) == [form] * len(calls), name


def test_no_early_tables():
    """A workspace of one sample's state and nothing else."""
    g = I.ba(29000, 3, seed=5)
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=8 * 8 * g.n)
    try:
        v = G.set_root()
        G.sample(12, 41)
        c1, c2, _ = G.counts()
        assert G.stat(LAP_STAT_LAST_FORM) == LAP_FORM_BLOCK
    finally:
        G.close()
    c = oracle.sample(g.row_ptr, g.col, v, 41, 0, 12)
    assert np.array_equal(c1, c.cnt1) and np.array_equal(c2, c.cnt2)


@pytest.mark.parametrize("option,form", [((LAP_OPT_KERNEL, 1), LAP_FORM_WIDE), ((LAP_OPT_KERNEL, 2), LAP_FORM_COMPACT),
                                         ((LAP_OPT_WALKERS, 8), LAP_FORM_GROUP)])
def test_options_take_their_kernel(option, form):
    assert form_of(I.ba(20000, 3, seed=1), [10], 1 << 26, [option]) == [form]


@pytest.mark.parametrize("kernel,form", [(0, LAP_FORM_BLOCK), (1, LAP_FORM_WIDE)])
def test_trees_take_their_kernel(kernel, form):
    g = I.ba(4097, 3, seed=2)
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=1 << 28)
    try:
        G.set_option(LAP_OPT_KERNEL, kernel)
        G.set_root()
        G.spantree_sample(200, 9)
        assert G.stat(LAP_STAT_TREE_FORM) == form
    finally:
        G.close()


def test_batches_take_branches():
    graphs = graphs20()
    B = LapBatch([(g.row_ptr, g.col) for g in graphs], workspace_bytes=1 << 30)
    try:
        B.run(24, 11)
        assert B.stat(LAP_BSTAT_BRANCHES) == len(graphs)
        B.set_option(LAP_BOPT_LANES, 40)
        B.run(24, 11)
        assert B.stat(LAP_BSTAT_BRANCHES) == 0
    finally:
        B.close()
