"""Device memory that a batch takes for packed arcs: 8 bytes for each arc of the graphs that
have them (96 MB at most per graph), none for larger graphs and none for a CSR that several
graphs of the batch share."""
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import LapBatch  # noqa: E402


def bytes_of(graphs):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    B = LapBatch([(g.row_ptr, g.col) for g in graphs], workspace_bytes=1 << 20)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    B.close()
    torch.cuda.empty_cache()
    return used


def test_packed_arcs_of_large_graphs():
    large = I.rmat(18, 32, seed=1)                       # too many arcs to be packed
    assert 8 * large.arcs > 96 << 20
    small = I.ba(100000, 10, seed=1)
    assert 8 * small.arcs <= 96 << 20
    bytes_of([small])                                    # (the library's own first allocations)
    alone, both, shared = bytes_of([large]), bytes_of([large, small]), bytes_of([large, small, small])
    # Column, packed arc and per-node arrays of the small graph, plus the allocator's granularity.
    assert both - alone < 12 * small.arcs + 200 * small.n + (24 << 20)
    assert shared - both < 200 * small.n + (24 << 20)
