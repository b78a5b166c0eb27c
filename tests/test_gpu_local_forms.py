"""mm_motor_local over the forms its rows take -- packed or a few nodes to a lane,
in registers by one warp and by several, in shared memory -- against the oracle,
to the tolerances of the local tests (float64 1e-12, float32 1e-5)."""
import numpy as np
import pytest

from paper_1908_04279_gb300.inputs import Grid, Rates
from tests.test_gpu_local import TOL, assert_close, count_margin, mmod, run_both, seeded  # noqa: F401

pytestmark = pytest.mark.gpu


# float64: few and short rows (two nodes to a lane, one), many (packed)
@pytest.mark.parametrize("dims", [(6, 5, 8, 8), (6, 5, 8, 7), (5, 4, 16, 8), (5, 4, 8, 16),
                                  (4, 3, 11, 13), (4, 3, 24, 30), (4, 3, 3, 1), (3, 3, 37, 64)])
def test_fp64_row_forms(mmod, oracle_mod, dims):  # noqa: F811
    g = Grid(*dims)
    psi, mb = seeded(g, 11 + sum(dims))
    st, gs, n_or, n_gpu = run_both(mmod, oracle_mod, g, Rates(), psi, mb, None, 0.37, "fp64")
    assert np.array_equal(n_gpu, n_or)
    assert_close(st, gs, TOL["fp64"], psi)
