"""A right-hand side that is not a number, or infinite, leaves no residual that a caller
could take for a solution; a zero one is solved exactly."""
import numpy as np
import pytest

from paper_2311_10290_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2311_10290_gb300.lap import LapGraph  # noqa: E402


@pytest.mark.parametrize("value", [float("nan"), float("inf"), 0.0])
def test_residual_of_a_bad_right_hand_side(value):
    g = I.ba(700, 3, seed=1)
    G = LapGraph(g.row_ptr, g.col, workspace_bytes=1 << 20)
    try:
        v = G.set_root()
        b = np.zeros(g.n)
        b[(v + 1) % g.n] = value
        x, it, res = G.lv_solve(b, rtol=1e-8, maxiter=20)
    finally:
        G.close()
    if value == 0.0:
        assert res == 0.0 and it == 0 and not np.any(x)
    else:
        assert not res <= 1e-8 and it == 20
