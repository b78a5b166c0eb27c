"""A resident launch that fails on the host (mm_debug_set makes the call return an
error instead of launching): the handle is as it was before the call, and the
next call works; a batch that had advanced in part says so and wants its states
set again."""
import numpy as np
import pytest

from paper_1908_04279_gb300.inputs import Grid, Rates, SplitMix64, psi_isotropic_perturbed, random_divfree_flow

pytestmark = pytest.mark.gpu

KEYS = ("psi", "mb", "mf", "c")


@pytest.fixture(scope="module")
def mmod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1908_04279_gb300 import build as B
    B.build()
    from paper_1908_04279_gb300 import mm
    mm.load_library()
    return mm


def set_up(sim, seed):
    g = sim.grid
    mb = 0.3 * SplitMix64(seed).uniforms(g.micro_cells).reshape(g.ny, g.nx, g.ntheta, g.ns)
    sim.set_state(psi_isotropic_perturbed(g, seed, amp=0.3), mb)
    sim.set_velocity(random_divfree_flow(g, seed + 1, 5, 0.15))


def test_failed_launch_leaves_the_handle(mmod):
    g = Grid(24, 20, 16, 16)
    got = []
    for fail in (False, True):
        with mmod.Simulation(g, Rates(), "fp32") as sim:
            set_up(sim, 3)
            sim.step(4)
            if fail:
                sim.debug_set(1 << 22, 1 << 8)
                with pytest.raises(mmod.MMError) as e:
                    sim.step(5)
                assert e.value.status == 3  # MM_ERR_CUDA
            sim.step(5)
            sim.sync()
            got.append(sim.get_state())
    for k in KEYS:
        assert np.array_equal(got[0][k], got[1][k]), k


def test_failed_group_launch(mmod):
    """Two members of 67 MB, a group (a launch) each."""
    grids = [Grid(128, 128, 32, 32)] * 2
    with mmod.Batch(grids, [Rates(), Rates(k_off=0.7)], "fp32") as b:
        want = None
        for first in (None, 1, 2):
            for i, sim in enumerate(b.members):
                set_up(sim, 5 + i)
            b.step(3)
            if first:
                b.debug_set(1 << 22, first << 8)
                with pytest.raises(mmod.MMError) as e:
                    b.step(3)
                assert e.value.status == 3
            if first == 2:  # the first member has advanced, the second has not
                with pytest.raises(mmod.MMError) as e:
                    b.step(3)
                assert e.value.status == 7  # MM_ERR_STATE
                for i, sim in enumerate(b.members):
                    set_up(sim, 5 + i)
                b.step(3)
            b.step(3)
            b.sync()
            got = [sim.get_state() for sim in b.members]
            want = want or got
            for a, c in zip(got, want):
                for k in KEYS:
                    assert np.array_equal(a[k], c[k]), (first, k)
