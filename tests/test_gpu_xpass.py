"""The binning x pass where its layout changes with the length, the fields and the bins: rows packed into
a warp, rows of several warps, rows that take whole 96-thread CTAs (3 * 2^k), partial sums in shared or
global memory, with and without interlacing, even and odd multipoles, a global line of sight."""
import numpy as np
import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import power as P  # noqa: E402
from synthetic import make_periodic_catalog, make_survey_catalogs  # noqa: E402
from helpers import ensure_built, p_error  # noqa: E402


@pytest.fixture(scope="module")
def api():
    ensure_built()
    from paper_2605_04864_gb300 import api as a

    return a


def _compare(res, orc, ells, modified, tol):
    scale = np.abs(orc["P"][0]) + orc["scalars"]["N0"] if 0 in orc["P"] else None
    assert np.array_equal(res["nmodes"], orc["nmodes"])
    for l in ells:
        assert np.max(p_error(res["P"][l], orc["P"][l], scale)) <= tol
    for l in modified:
        assert np.max(p_error(res["Pmod"][l], orc["Pmod"][l], scale)) <= tol


# 300 narrow bins: partial sums too large for shared memory, many of them empty
@pytest.mark.parametrize("nbins", [9, 300])
@pytest.mark.parametrize("interlace", [0, 1])
@pytest.mark.parametrize("n,prec,tol", [(16, "fp64", 1e-12), (32, "mixed", 1e-5), (48, "mixed", 1e-5), (64, "fp64", 1e-12)])
def test_all_multipoles(api, n, prec, tol, interlace, nbins):
    box, dtype = 500.0, np.float64 if prec == "fp64" else np.float32
    g, r, o = make_survey_catalogs(3_001, 20_011, box, 900.0, 16, seed=n + interlace, fkp_p0=1e4, dtype=dtype)
    kb = (0.0, 0.5 * np.pi * n / box / nbins * 2.2, nbins)
    ells, mod = (0, 1, 2, 3, 4), (4, 6, 8)
    spec = dict(n=n, box=box, origin=tuple(o), assign=3, interlace=interlace, los="endpoint", observer=(0.0, 0.0, 0.0))
    res = api.power_multipoles(g, r, n=n, box=box, origin=o, interlace=interlace, kbins=kb, ells=ells, modified=mod,
                               precision=prec)
    _compare(res, P.power_multipoles(spec, g, r, kb, ells, mod), ells, mod, tol)


@pytest.mark.parametrize("nbins", [7, 300])
@pytest.mark.parametrize("n,prec,tol", [(16, "mixed", 1e-5), (48, "fp64", 1e-12), (64, "mixed", 1e-5)])
def test_global_line_of_sight(api, n, prec, tol, nbins):
    """Rows ky and -ky are binned together; a tilted line of sight tells their modes apart."""
    box = 300.0
    c = make_periodic_catalog(4_003, box, 16, seed=n, dtype=np.float64 if prec == "fp64" else np.float32)
    kb = (0.0, np.pi * n / box / nbins * 1.1, nbins)
    ells, los = (0, 1, 2, 3, 4), (0.3, -0.5, 0.8)
    spec = dict(n=n, box=box, origin=(0.0, 0.0, 0.0), assign=3, interlace=1, los="global", los_dir=los, periodic=1)
    res = api.power_multipoles(c, None, n=n, box=box, kbins=kb, ells=ells, modified=(4,), precision=prec, los_dir=los)
    _compare(res, P.power_multipoles(spec, c, None, kb, ells, (4,)), ells, (4,), tol)
