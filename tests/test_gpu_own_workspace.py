"""The workspace that a handle allocates itself, where none is lent: what the lanes of the
call's kernel can use, whichever sampler the call takes."""
import pytest

import oracle
from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300 import lap  # noqa: E402


@pytest.mark.parametrize("kernel,slot", [(0, 1024 + 4 * 1024 + 8 * 1024), (1, 8 * 1000)], ids=["automatic", "wide"])
def test_bytes_of_own_workspace(kernel, slot):
    g = I.ba(1000, 3, seed=1)
    torch.zeros(1, device="cuda")
    h = lap.lap_graph_create(g.n, g.row_ptr, g.col)
    try:
        lap.lap_set_option(h, lap.LAP_OPT_KERNEL, kernel)
        v = lap.lap_set_root(h)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        lap.lap_sample(h, 100, 7)
        lap.lap_sync(h)
        used = before - torch.cuda.mem_get_info()[0]
        c1, c2, sums = lap.lap_counts(h, g.n)
    finally:
        lap.lap_graph_destroy(h)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert used < slot * sms * 2048 + (64 << 20)          # (tables of a few bytes per sample beside it)
    c = oracle.sample(g.row_ptr, g.col, v, 7, 0, 100, keep_per_sample=False)
    assert (c1 == c.cnt1).all() and (c2 == c.cnt2).all()
