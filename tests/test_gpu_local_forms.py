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


# float32 cells of several warps in registers: 10 and 16 (the most), ragged rows, and
# a cell of more row passes than registers take (the shared-memory kernel)
WIDE = [(3, 2, 160, 64), (2, 2, 512, 32), (3, 2, 200, 30), (2, 2, 320, 64)]


@pytest.mark.parametrize("dims", WIDE)
def test_fp32_wide_cells(mmod, oracle_mod, dims):  # noqa: F811
    g = Grid(*dims)
    r = Rates(v_walk=0.09)
    psi, mb = seeded(g, 61 + sum(dims))
    T = next(t for t in (2.41, 2.43, 2.47, 2.53, 2.59, 2.61) if count_margin(g, r, psi, t) > 1e-4)
    st, gs, n_or, n_gpu = run_both(mmod, oracle_mod, g, r, psi, mb, None, T, "fp32")
    assert np.array_equal(n_gpu, n_or)
    assert_close(st, gs, TOL["fp32"], psi)


@pytest.mark.parametrize("dims", WIDE)
def test_fp32_wide_cells_scale_down(mmod, oracle_mod, dims):  # noqa: F811
    g = Grid(*dims)
    psi, mb = seeded(g, 41, mb_scale=0.05)
    mtot = 0.1 * np.ones((g.ny, g.nx))
    nsteps = (1 + np.arange(g.ncells) % 3).reshape(g.ny, g.nx).astype(np.int32)
    st, gs, _, n_gpu = run_both(mmod, oracle_mod, g, Rates(k_on=40.0, k_off=0.1), psi, mb, mtot,
                                0.5, "fp32", nsteps)
    assert np.array_equal(n_gpu, nsteps)
    assert np.all(np.abs(st.c - mtot)[nsteps == 1] == 0)  # the scale-down was taken
    assert_close(st, gs, TOL["fp32"], psi)


def test_fp32_shared_memory_timeout(mmod, oracle_mod):  # noqa: F811
    """The knob on: the shared-memory kernel's bounded waits run out, its copies are
    drained and the call says so; then the same handle gives the oracle's answer."""
    g = Grid(2, 2, 320, 64)
    psi, mb = seeded(g, 91)
    T = next(t for t in (0.2, 0.21, 0.22, 0.23) if count_margin(g, Rates(), psi, t) > 1e-4)
    with mmod.Simulation(g, Rates(), "fp32") as sim:
        sim.set_state(psi, np.ascontiguousarray(mb))
        sim.debug_set(2000, 1)
        with pytest.raises(mmod.MMError) as e:
            sim.motor_local(T)
        assert e.value.status == 5
        sim.debug_set(1 << 22, 0)
        sim.set_state(psi, np.ascontiguousarray(mb))
        n_gpu = sim.motor_local(T)
        gs = sim.get_state()
    st = oracle_mod.make_state(g, psi, mb)
    assert np.array_equal(n_gpu, oracle_mod.motor_local(g, Rates(), st, T))
    assert_close(st, gs, TOL["fp32"], psi)
