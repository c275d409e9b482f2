"""The 32-bit words of a tile sum when they overflow: objects that lie on grid points, so that every tap is
an exact integer in the tile's fixed point and the integer parts add up coherently."""
import numpy as np
import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_paint import _paint  # noqa: E402

N = 48   # bricks of 16 cells
EPS = 2.0**-24


def _parts(w, cnt):
    """The kernel's split of a whole tap: w 2^e = 2^22 h + l with both |h|, |l| <= 2^21."""
    mant, ex = np.frexp(float(cnt) * float(np.abs(w).max()))
    e = min((60 if mant > 127 / 128 else 61) - ex, 43 - np.frexp(float(np.abs(w).max()))[1])
    v = w.astype(np.float64) * 2.0**e
    h = np.rint(v / 2.0**22)
    return h, v - h * 2.0**22


def _objects(cells, weights, counts):
    pos = np.repeat(np.asarray(cells, np.float32), counts, axis=0)
    return pos, np.repeat(np.asarray(weights, np.float32), counts)


def _check(pos, w, cells, weights, counts):
    """CIC at grid points: each object's weight falls on its cell.  The cell's sum is exact until it is rounded
    to float32 once per word, the mean is subtracted and the result is rounded: 4 x 2^-24 of the cell."""
    got = _paint(pos, w, N, float(N), 2)
    want = np.zeros((N, N, N))
    for c, x, m in zip(cells, weights, counts):
        want[c] += float(np.float32(x)) * m
    mean = want.sum() / N**3
    assert np.all(np.abs(got - (want - mean)) <= 4 * EPS * np.abs(want) + 2 * EPS * abs(mean))


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("count", [1023, 1024, 1025, 2047, 2049])
def test_low_word(count, sign):
    """Weights 1 + 2^-21 leave l = 2^21 each: the sum reaches 2^31 at 1024 objects.  A lost carry is 2^-10 of
    a weight, far above the 4 x 2^-24 of these sums."""
    w = np.float32(sign * (1 + 2.0**-21))
    _, low = _parts(np.array([w]), count)
    assert abs(low[0]) == 2**21 and (count < 1024 or abs(low[0]) * count >= 2**31 - (sign < 0))
    assert 4 * EPS * count * 1.001 < 2.0**-10   # the bound of the sum is below a lost carry
    cells = [(17, 20, 21)]
    pos, wt = _objects(cells, [w], [count])
    _check(pos, wt, cells, [w], [count])


@pytest.mark.parametrize("pattern", [(1, 1, 1, 1), (-1, -1, -1, -1), (1, -1, 1, -1), (-1, 1, 1, -1), (-1, 0, 0, 1)])
def test_high_words_of_neighbours(pattern):
    """Weights just below 2 give h = 2^21 each: 16,383 objects wrap a cell's high word about eight times,
    either way, and x neighbours keep their digits in the bytes of one word, which borrow from one another.
    A lost digit is 2^12 weights."""
    w = 2.0 - 2.0**-22
    cells = [(16 + i, 18, 19) for i in range(8)]
    weights = [s * w for s in pattern + pattern[::-1]]
    counts = [16_383 if s else 0 for s in pattern + pattern[::-1]]
    high, _ = _parts(np.array([w], np.float32), sum(counts))
    assert high[0] * counts[0] >= 7.9 * 2**32
    pos, wt = _objects(cells, weights, counts)
    order = np.random.default_rng(1).permutation(len(wt))
    _check(pos[order], wt[order], cells, weights, counts)


def test_high_word_of_both_signs():
    """Positive and negative objects of one cell in two runs: the word wraps up and down again."""
    w = 2.0 - 2.0**-22
    cells, weights, counts = [(33, 34, 35), (33, 34, 35), (36, 34, 35)], [w, -w, w], [20_000, 16_000, 3_000]
    pos, wt = _objects(cells, weights, counts)
    _check(pos, wt, cells, weights, counts)


def test_smallest_unit_of_a_full_brick():
    """300,000 objects of weights +1 and -1 in a brick (2^18 < 300,000 < 2^19) leave 2^-42 as the unit of the
    tile's sums: a lone weight of 2^-42 keeps its value.  With a unit of 2^-41 it is a tie and rounds to 0."""
    cells, weights, counts = [(2, 2, 2), (5, 2, 2), (9, 9, 9)], [1.0, -1.0, 2.0**-42], [150_000, 150_000, 1]
    pos, wt = _objects(cells, weights, counts)
    got = _paint(pos, wt, N, float(N), 2)
    assert abs(got[9, 9, 9] - 2.0**-42) <= 2.0**-42 * 2.0**-10


@pytest.mark.parametrize("cells,count", [([(3, 3, 3)], 262_144), ([(3, 3, 3), (4, 3, 3)], 131_072), ([(3, 3, 3)], 260_000)])
@pytest.mark.parametrize("sign", [1, -1])
def test_fullest_cells(cells, count, sign):
    """Weights just below 2 on one or two points, bounds on either side of 127/128 of a power of two: the digits
    of the high word come to +-64 and +-127."""
    w = sign * (2.0 - 2.0**-22)
    weights = [w, -w][: len(cells)]
    pos, wt = _objects(cells, weights, [count] * len(cells))
    _check(pos, wt, cells, weights, [count] * len(cells))
