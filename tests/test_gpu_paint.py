"""Painting kernels at the sizes where their paths change, against the oracle's float64 assignment."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mesh as OM  # noqa: E402

EPS = 2.0**-24


def _paint(pos, w, n, box, assign):
    from paper_2605_04864_gb300 import autograd

    m = autograd.paint(torch.tensor(pos, device="cuda"), torch.tensor(w, device="cuda"), n, box, assign=assign)
    return m.cpu().numpy().transpose(2, 1, 0)   # the mesh is indexed z, y, x


def _check(pos, w, n, box, assign, per_cell):
    """per_cell: sum of |w| over the objects that can reach a cell.  A tap's three weights are each off
    by at most 2^-24 of a cell times a slope <= 1 plus a rounding, so a cell by 6 x 2^-24 per object;
    the sum of the tiles and the mean add 2^-22 of the cell and 2^-23 of the mean."""
    got = _paint(pos, w, n, box, assign)
    wd = w.astype(np.float64)
    painted = OM.paint(OM.grid_coords(pos, np.zeros(3), box, n), wd, n, assign)
    mean = float(wd.sum()) / n**3
    bound = 6 * EPS * per_cell * (painted != 0) + 4 * EPS * np.abs(painted) + 2 * EPS * abs(mean)
    assert np.all(np.abs(got - (painted - mean)) <= bound)


@pytest.mark.parametrize("assign", [2, 3])
@pytest.mark.parametrize("nobj", [1, 1023, 1024, 2428, 5200])
@pytest.mark.parametrize("sign", ["positive", "negative", "mixed"])
def test_tile_words_carry(nobj, assign, sign):
    """All objects in one cell: the low words of a tile sum can overflow from 1024 objects on, the high
    ones from about 2427.  A lost carry of the high word is 2^12 largest weights, of the low one 2^-10."""
    rng = np.random.default_rng(nobj)
    pos = (np.array([7.0, 8.0, 15.0]) + rng.random((nobj, 3))).astype(np.float32)
    w = (rng.random(nobj) + 0.5).astype(np.float32)
    if sign != "positive":
        w *= np.where((rng.random(nobj) < 0.5) | (sign == "negative"), -1, 1).astype(np.float32)
    _check(pos, w, 32, 32.0, assign, float(np.abs(w).sum()))
