"""iwf_evaluate_grid at the edges of its tiles (128 rows x 64 columns, whose rows and columns are
summed in pairs around the tile's centre): single points, odd and even remainders, a negative
and an uneven step, against the oracle's direct sum.

Tolerance: that of iwf_evaluate's tests. The centre's phase and the pair's phase together are no
larger than the point's, each rounded to eps of itself; a pair's point differs from
origin + index * step by that coordinate's own rounding (eps |x|, a phase of eps |theta|).
"""
import numpy as np
import pytest

from oracle import transform as T

from test_gpu_evaluate import GRID_PROBS, _grid_points, _setup, _tol

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["moire_ragged", "ex42"])
@pytest.mark.parametrize("count", [(1, 1), (2, 63), (127, 64), (128, 65), (129, 2), (257, 1)])
def test_tile_edges_match_oracle(name, count):
    import paper_2404_04507_gb300 as iwf
    plan, win, c = _setup(iwf, GRID_PROBS[name])
    origin, step = (17.25, -40.0), (-0.3, 0.07)
    got = plan.evaluate_grid(torch.from_numpy(c).cuda(), origin, step, count)
    x = _grid_points(origin, step, count)
    want = T.evaluate_quasi(win, c, x)
    assert np.max(np.abs(got.cpu().numpy() - want)) <= _tol(win, c, x)
