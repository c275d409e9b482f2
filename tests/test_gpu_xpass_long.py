"""The binning x pass on the longest rows, which take several warps each: at 512 an even number of exchanges
per transform, at 1024 an odd one (the two exchange buffers change places from row to row), with and without
the rows ky and -ky binned together.  Few objects and bins; the reference is the float64 evaluation of the
performance cases, plain torch transforms on the same catalogue."""
import importlib.util
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from helpers import ROOT, ensure_built, p_error  # noqa: E402


@pytest.fixture(scope="module")
def cases():
    ensure_built()
    spec = importlib.util.spec_from_file_location("cases", os.path.join(ROOT, "perf", "cases.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.mark.parametrize("n,n_ran,interlace,ells,nbins", [
    (512, 200_010, 0, "0,1,2,3,4", 12),
    (512, 200_010, 1, "0,2", 50),
    (512, 0, 1, "0,2,4", 50),
    (1024, 200_010, 0, "0,2", 12),
    (1024, 0, 1, "0,1,2,4", 30),
])
def test_rows_of_several_warps(cases, n, n_ran, interlace, ells, nbins):
    case = cases._power(n, 2000.0, 20_001, n_ran, nbins, ells=ells, interlace=interlace)
    got = {k: v.double().cpu().numpy() for k, v in cases.run(cases.prepare(case, 3)).items()}
    want = {k: v.cpu().numpy() for k, v in cases.exact(case, 3).items()}
    assert np.array_equal(got["nmodes"], want["nmodes"])
    scale = np.abs(want["P0"]) + want["scalars"][3]
    for l in ells.split(","):
        assert np.max(p_error(got["P" + l], want["P" + l], scale)) <= 1e-5, l
