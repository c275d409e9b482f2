"""The transform autotuner: it times the kernels that measurements launch, and no choice changes a result."""
import numpy as np
import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from synthetic import make_survey_catalogs  # noqa: E402
from helpers import ensure_built  # noqa: E402


@pytest.mark.parametrize("n,prec,plain,weighted", [
    (16, "mixed", 3, 3), (48, "fp64", 3, 3), (64, "mixed", 4, 4), (192, "fp64", 4, 4),
    (256, "fp64", 4, 3),    # 32 float64 columns and their copy do not fit
    (512, "mixed", 3, 3),
])
def test_times_both_forms_of_the_y_pass(n, prec, plain, weighted):
    """A warm-up and three timed launches per width, of the plain pass and of the one with column factors."""
    ensure_built()
    from paper_2605_04864_gb300 import api

    g, r, origin = make_survey_catalogs(2_000, 10_000, 500.0, 900.0, 16, seed=n, fkp_p0=1e4)

    def run():
        return api.power_multipoles(g, r, n=n, box=500.0, origin=origin, kbins=(0.0, 0.02, 6), ells=(0, 2, 4),
                                    precision=prec)["P"]

    before = run()
    api.tune_transforms(n, prec)
    assert api.last_stats()["n_kernel_launches"] == 4 * (plain + weighted)
    after = run()
    for ell in (0, 2, 4):
        assert np.array_equal(before[ell], after[ell])
