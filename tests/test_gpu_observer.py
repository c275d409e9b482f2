"""Directions from an observer among the grid points, or in large or small units of length: the signals of
the weighted first passes stay finite and match the oracle where a grid point lies at the observer up to
the rounding of its coordinates, and for any scale of the coordinates."""
from types import SimpleNamespace

import numpy as np
import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import bispec as OB  # noqa: E402
from oracle import power as P  # noqa: E402
from oracle import sugiyama as OS  # noqa: E402
from synthetic import make_survey_catalogs  # noqa: E402
from helpers import ensure_built, p_error  # noqa: E402

NEXT = float(np.nextafter(512.7, 1e3))   # the origin plus half a box of 1000 misses it by one rounding


@pytest.fixture(scope="module")
def api():
    ensure_built()
    from paper_2605_04864_gb300 import api as a

    return a


def _around(observer, origin, box, cell, dtype, nd=4_001, nr=30_011):
    """Objects over the box, one in twenty of them within a cell of the observer."""
    rng = np.random.default_rng(11)

    def cat(m, nbar):
        pos = np.asarray(origin) + rng.random((m, 3)) * box
        near = rng.random(m) < 0.05
        pos[near] = np.asarray(observer) + (rng.random((near.sum(), 3)) - 0.5) * 2 * cell
        w = rng.random(m) * 0.5 + 0.5
        return SimpleNamespace(pos=pos.astype(dtype), w=w.astype(dtype), nbar=np.full(m, nbar, dtype))

    return cat(nd, nd / box**3), cat(nr, nd / box**3)


def _spec(n, box, origin, observer, interlace, **kw):
    return dict(n=n, box=box, origin=tuple(origin), assign=3, interlace=interlace, los="endpoint",
                observer=tuple(observer), **kw)


# the errors of the existing comparisons: 1e-5 of the monopole in mixed precision, 1e-12 in float64
@pytest.mark.parametrize("prec,tol", [("mixed", 1e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("interlace", [0, 1])
@pytest.mark.parametrize("n,box,origin,observer", [
    (48, 500.0, (-250.0,) * 3, (0.0,) * 3),                   # box/n inexact, a grid point exactly at the observer
    (32, 1000.0, (12.7,) * 3, (NEXT,) * 3),                   # a grid point 1e-13 off on every axis
    (32, 1000.0, (12.7,) * 3, (NEXT, 512.7, 300.0)),          # grid lines along y and z through the observer
    (32, 1000.0, (-484.375, -484.375, -900.0), (0.0,) * 3),   # a column of the shifted phase through the observer
    (32, 1000.0, (-507.99, -507.99, -500.0), (0.0,) * 3),     # a column within the 8 that count as near ...
    (32, 1000.0, (-508.01, -507.99, -500.0), (0.0,) * 3),     # ... and none
])
def test_multipoles_with_the_observer_on_a_grid_line(api, n, box, origin, observer, interlace, prec, tol):
    g, r = _around(observer, origin, box, box / n, np.float64 if prec == "fp64" else np.float32)
    kb = (0.0, 0.2 * np.pi * n / box, 5)
    ells, mod = (0, 1, 2, 3, 4), (4, 6, 8)
    res = api.power_multipoles(g, r, n=n, box=box, origin=origin, observer=observer, interlace=interlace, kbins=kb,
                               ells=ells, modified=mod, precision=prec)
    orc = P.power_multipoles(_spec(n, box, origin, observer, interlace), g, r, kb, ells, mod)
    scale = np.abs(orc["P"][0]) + orc["scalars"]["N0"]
    for l in ells:
        assert np.max(p_error(res["P"][l], orc["P"][l], scale)) <= tol, l
    for l in mod:
        assert np.max(p_error(res["Pmod"][l], orc["Pmod"][l], scale)) <= tol, l


@pytest.mark.parametrize("interlace", [0, 1])
@pytest.mark.parametrize("unit", [2.0**34, 2.0**-34, 1e10])
def test_units_of_length(api, unit, interlace):
    """All lengths in another unit, far above and below that of the catalogues."""
    n, box = 32, 500.0 * unit
    g, r, o = make_survey_catalogs(3_001, 20_011, 500.0, 900.0, 16, seed=5, fkp_p0=1e4, dtype=np.float64)
    ells, kb, o = (0, 1, 2, 3, 4), (0.0, 0.02 / unit, 9), tuple(np.asarray(o) * unit)

    def scaled(c):
        return SimpleNamespace(pos=(c.pos * unit).astype(np.float32), w=np.asarray(c.w).astype(np.float32),
                               nbar=(c.nbar / unit**3).astype(np.float32))

    g, r = scaled(g), scaled(r)
    res = api.power_multipoles(g, r, n=n, box=box, origin=o, interlace=interlace, kbins=kb, ells=ells,
                               precision="mixed")
    orc = P.power_multipoles(_spec(n, box, o, (0.0,) * 3, interlace), g, r, kb, ells)
    scale = np.abs(orc["P"][0]) + orc["scalars"]["N0"]
    for l in ells:
        assert np.max(p_error(res["P"][l], orc["P"][l], scale)) <= 1e-5, l


@pytest.mark.parametrize("observer", [(0.0,) * 3, (2.0**-44,) * 3])
def test_odd_bispectrum_multipoles(api, observer):
    n, box, origin = 48, 500.0, (-250.0,) * 3
    g, r = _around(observer, origin, box, box / n, np.float32)
    kf = 2 * np.pi / box
    kb = (2 * kf, 2 * kf, 3)
    res = api.bispectrum(g, n=n, box=box, kbins=kb, precision="mixed", origin=origin, randoms=r, los_dir=None,
                         observer=observer, scoc_ells=(0, 1, 3), tripo_ells=(0,))
    orc = OB.odd_multipoles(_spec(n, box, origin, observer, 1, periodic=0), g, r, kb, (1, 3))
    scale = np.abs(res["B"][0] + res["shot_B"][0])
    for l in (1, 3):
        assert np.max(np.abs(res["B"][l] - orc["B"][l]) / np.maximum(np.abs(orc["B"][l]), scale)) <= 1e-4, l


@pytest.mark.parametrize("corner", [-250.0, float(np.nextafter(-250.0, -1e3))])
def test_endpoint_tripolar_multipoles(api, corner):
    n, box, origin, observer = 48, 500.0, (corner,) * 3, (0.0,) * 3
    multipoles = [(0, 0, 0), (2, 1, 3)]
    g, r = _around(observer, origin, box, box / n, np.float32)
    kf = 2 * np.pi / box
    kb = (2 * kf, 2 * kf, 3)
    res = api.bispectrum_sugiyama(g, n=n, box=box, kbins=kb, multipoles=multipoles, los_dir=None, precision="mixed",
                                  origin=origin, randoms=r)
    spec = _spec(n, box, origin, observer, 1, periodic=0)
    sc = P.catalog_scalars(g, r, box)
    orc = OS.sugiyama_fft(spec, P.fkp_meshes(spec, g, r, sc), kb, multipoles, sc["I33"])
    scale = np.abs(np.real(orc[(0, 0, 0)]))
    for mp in multipoles:
        want = np.imag(orc[mp]) if (mp[0] + mp[1]) % 2 else np.real(orc[mp])
        assert np.max(np.abs(res["B"][mp] - want) / np.maximum(np.abs(want), scale)) <= 1e-4, mp
