"""Calls of one substep, which go to the streaming kernels whatever the size: the
float32 batch over tiles (units of one cell and of two, before and after the
autotuner) against the oracle and the members alone, and the bounded waits and
drains of both streaming kernels in float32, which longer calls no longer reach."""
import numpy as np
import pytest

from paper_1908_04279_gb300.inputs import Grid, Rates, cellular_flow, member_inputs, psi_isotropic_perturbed
from tests.test_gpu_batch import alone, members, mmod, rel, setup  # noqa: F401

pytestmark = pytest.mark.gpu

KEYS = ("psi", "mb", "mf", "c")


@pytest.mark.parametrize("tuned", [False, True])
def test_float32_batch_over_tiles(mmod, oracle_mod, tuned):  # noqa: F811
    ms = members()
    with mmod.Batch([m.grid for m in ms], [m.rates for m in ms], "fp32") as b:
        setup(b, ms)
        if tuned:
            b.autotune(substeps=2)
        dts = [s.dt for s in b.members]
        for i in range(9):
            if i == 4:
                b.members[1].step(1)  # one member alone: parities diverge
            b.step(1)
        b.sync()
        states = [s.get_state() for s in b.members]
    for i, m in enumerate(ms):
        n = 9 + (i == 1)
        st = alone(mmod, m, "fp32", [1] * n)
        psi0, u = member_inputs(m, modes=4, amp=0.3)
        o = oracle_mod.make_state(m.grid, psi0)
        oracle_mod.run(m.grid, m.rates, o, u, dts[i], n)
        for k in ("psi", "mb", "mf"):
            assert rel(states[i][k], getattr(o, k)) <= 1e-5, (i, k)
            assert rel(states[i][k], st[k]) <= 1e-6, (i, k)


@pytest.mark.parametrize("ns", [32, 28, 30])
def test_streaming_timeout(mmod, ns):  # noqa: F811
    g = Grid(16, 16, 32, ns)
    psi, u = psi_isotropic_perturbed(g, 0), cellular_flow(g)
    got = []
    for knob in (False, True):
        with mmod.Simulation(g, Rates(), "fp32") as sim:
            assert sim.launch_info()["tma"] == 1
            sim.set_state(psi)
            sim.set_velocity(u)
            if knob:
                sim.debug_set(2000, 1)
                sim.step(1)
                with pytest.raises(mmod.MMError) as e:
                    sim.sync()
                assert e.value.status == 5  # MM_ERR_TIMEOUT
                sim.debug_set(1 << 22, 0)
                sim.set_state(psi)
                sim.set_velocity(u)
            for _ in range(3):
                sim.step(1)
            sim.sync()
            got.append(sim.get_state())
    for k in KEYS:
        assert np.array_equal(got[0][k], got[1][k]), k


def test_batch_tiles_timeout(mmod):  # noqa: F811
    ms = members()
    got = []
    for knob in (False, True):
        with mmod.Batch([m.grid for m in ms], [m.rates for m in ms], "fp32") as b:
            setup(b, ms)
            if knob:
                b.debug_set(64, 1)
                b.step(1)
                with pytest.raises(mmod.MMError) as e:
                    b.sync()
                assert e.value.status == 5
                b.debug_set(1 << 22, 0)
                setup(b, ms)
            for _ in range(3):
                b.step(1)
            b.sync()
            got.append([s.get_state() for s in b.members])
    for x, y in zip(*got):
        for k in KEYS:
            assert np.array_equal(x[k], y[k]), k
