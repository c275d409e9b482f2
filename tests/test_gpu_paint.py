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


@pytest.mark.parametrize("n", [16, 32, 96, 256])
@pytest.mark.parametrize("nobj", [1, 4095, 4096, 4097, 30_011])
def test_brick_sort_and_wrap(n, nobj):
    """Object numbers around the counting chunk, positions in cell order and up to two boxes outside:
    every object must reach its cells (4, 4, 6 and 16 bricks a side)."""
    rng = np.random.default_rng(n + nobj)
    pos = ((rng.random((nobj, 3)) * 5 - 2) * n).astype(np.float32)
    pos[: nobj // 2] = pos[np.lexsort(np.floor(pos[: nobj // 2]).T)]
    w = (rng.random(nobj) + 0.5).astype(np.float32)
    # reach of a cell: all objects within 3 cells of it, bounded by the densest 5^3 block
    cells = np.floor(pos.astype(np.float64)).astype(np.int64) % n
    dense = np.bincount((cells // 4) @ np.array([1, n, n * n]), weights=w).max()
    _check(pos, w, n, float(n), 3, 8.0 * dense)


def test_more_bricks_than_shared_counters():
    """512^3 has 32,768 bricks: per-object counters and a scan over several chunks.  Each of 5,003
    objects sits alone on a grid point, so its cell holds its weight and its neighbours known taps."""
    n, nobj = 512, 5_003
    rng = np.random.default_rng(5)
    cells = np.unique(rng.integers(0, 128, (nobj, 3)) * 4, axis=0)
    w = (rng.random(len(cells)) + 0.5).astype(np.float32)
    got = _paint(cells.astype(np.float32), w, n, float(n), 2)
    mean = float(w.astype(np.float64).sum()) / n**3
    at = got[cells[:, 0], cells[:, 1], cells[:, 2]]
    assert np.all(np.abs(at - (w - mean)) <= 6 * EPS * w)
    got[cells[:, 0], cells[:, 1], cells[:, 2]] = -mean
    assert np.all(np.abs(got + mean) <= 6 * EPS)


@pytest.mark.parametrize("swap", [False, True])
def test_catalogues_of_two_types(swap):
    """Data and randoms of different float types are sorted by two launches, of one type by one: the
    same positions give the same multipoles (to the rounding of the fractions and weights, 2^-20 of the
    monopole's scale)."""
    from types import SimpleNamespace

    from paper_2605_04864_gb300 import api

    rng = np.random.default_rng(3)
    def cat(m):
        return SimpleNamespace(pos=(rng.random((m, 3)) * 64 + 100).astype(np.float32), w=np.ones(m, np.float32),
                               nbar=np.full(m, 1e-2, np.float32))
    def wide(c):
        return SimpleNamespace(pos=c.pos.astype(np.float64), w=c.w.astype(np.float64), nbar=c.nbar.astype(np.float64))
    g, r = cat(2_000), cat(20_001)
    kw = dict(n=32, box=64.0, origin=(100.0,) * 3, kbins=(0.05, 0.1, 12))
    one = api.power_multipoles(g, r, **kw)
    two = api.power_multipoles(wide(g) if swap else g, r if swap else wide(r), **kw)
    scale = np.abs(one["P"][0]) + one["scalars"]["N0"]
    for ell in (0, 2, 4):
        assert np.all(np.abs(one["P"][ell] - two["P"][ell]) <= 2.0**-20 * scale)
