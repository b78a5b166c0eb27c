"""Many substeps in one launch with the motor density resident on the chip
(float32 form), against the float64 oracle (relative L2 1e-5, the float32
tolerance of the parity tests) and against the same handle stepped one substep
per call, which takes the streaming kernel (1e-6: the two differ in the order
of a few float32 sums)."""
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


def rel_l2(a, b):
    nb = np.linalg.norm(b)
    return np.linalg.norm(np.asarray(a, dtype=np.float64) - b) / (nb if nb > 0 else 1.0)


def inputs(g, seed, scale):
    rng = SplitMix64(seed)
    mb = scale * rng.uniforms(g.micro_cells).reshape(g.ny, g.nx, g.ntheta, g.ns)
    return psi_isotropic_perturbed(g, seed, amp=0.3), mb, random_divfree_flow(g, seed + 1, 5, 0.15)


# (grid, substeps, k_on): rows that end in every node of a lane and rows of one
# node; passes that span cells (few orientations) and orientations beyond a
# warp; fewer cells than SMs, several cells per warp; binding fast enough for
# the scale-down to act in the substeps (dt is then the one without it)
@pytest.mark.parametrize("dims,n,k_on", [
    ((6, 5, 7, 1), 4, 1.0), ((9, 7, 5, 31), 5, 1.0), ((7, 6, 20, 25), 4, 1.0),
    ((13, 11, 12, 10), 7, 1.0), ((5, 4, 40, 20), 4, 1.0), ((4, 3, 70, 36), 3, 1.0),
    ((3, 2, 6, 128), 4, 1.0), ((1, 1, 8, 16), 6, 1.0), ((40, 31, 16, 16), 5, 1.0),
    ((40, 40, 8, 9), 4, 1.0), ((45, 40, 24, 30), 4, 1.0), ((24, 20, 32, 32), 3, 1.0),
    ((20, 17, 16, 24), 6, 400.0), ((19, 16, 10, 13), 5, 400.0)])
def test_resident_substeps(mmod, dims, n, k_on):
    from oracle import oracle as O
    g = Grid(*dims)
    r = Rates(glide=0.3, v_sp=0.05, k_on=k_on)
    psi, mb, u = inputs(g, 11, 0.3)
    st = O.make_state(g, psi, mb)
    dt = O.dt(g, Rates(glide=0.3, v_sp=0.05), st, u)
    got = []
    for each in (n, 1):
        with mmod.Simulation(g, r, "fp32") as sim:
            sim.set_state(psi, mb)
            sim.set_velocity(u)
            sim.set_dt(dt)
            for _ in range(n // each):
                sim.step(each)
            got.append(sim.get_state())
            _, sc = sim.moments()
            assert abs(sc["N_psi"] - 1.0) < 1e-6  # the mass correction
    clipped = False
    for _ in range(n):
        O.run(g, r, st, u, dt, 1)
        clipped = clipped or st.mf.min() == 0.0
    assert clipped == (k_on > 1)  # where the scale-down acts
    for k in KEYS:
        assert rel_l2(got[0][k], getattr(st, k)) <= 1e-5, k
        assert rel_l2(got[0][k], got[1][k]) <= 1e-6, k


def test_resident_on_two_streams(mmod):
    """Two handles stepped alternately on two streams: the launches share the
    device one after the other and each result is that of a handle alone."""
    import torch
    g = Grid(48, 40, 16, 16)
    psi, mb, u = inputs(g, 3, 0.3)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for alternate in (False, True):
        sims = [mmod.Simulation(g, Rates(k_off=0.5 + i), "fp32", stream=s.cuda_stream)
                for i, s in enumerate(streams)]
        for sim in sims:
            sim.set_state(psi, mb)
            sim.set_velocity(u)
        order = [(i, n) for n in (30, 31, 32) for i in (0, 1)]
        for i, n in order if alternate else sorted(order):
            sims[i].step(n)
        got.append([sim.get_state() for sim in sims])
        for sim in sims:
            sim.close()
    for a, b in zip(*got):
        for k in KEYS:
            assert np.array_equal(a[k], b[k]), k


# rows kept in part: whole vectors, halves and single values of 16-byte copies,
# a grid a block of which holds cells of several rows
@pytest.mark.parametrize("dims", [(130, 96, 40, 24), (128, 128, 32, 32), (150, 120, 24, 30),
                                  (141, 130, 23, 29), (120, 110, 48, 36)])
def test_partly_kept_rows(mmod, dims):
    """Instances beyond the chip: the substeps of one call against one substep
    per call, and the conserved sums."""
    g = Grid(*dims)
    psi, mb, u = inputs(g, 7, 0.3)
    got = []
    for each in (5, 1):
        with mmod.Simulation(g, Rates(glide=0.3), "fp32") as sim:
            sim.set_state(psi, mb)
            sim.set_velocity(u)
            for _ in range(5 // each):
                sim.step(each)
            got.append(sim.get_state())
            _, sc = sim.moments()
            assert abs(sc["N_psi"] - 1.0) < 1e-6 and abs(sc["motors"] - 1.0) < 1e-5
    for k in KEYS:
        assert rel_l2(got[0][k], got[1][k]) <= 1e-6, k


def test_partly_kept_rows_scale_down(mmod):
    """The scale-down on rows that are not kept, against the oracle."""
    from oracle import oracle as O
    g = Grid(120, 110, 32, 24)
    r = Rates(k_on=400.0)
    psi, mb, u = inputs(g, 5, 0.3)
    st = O.make_state(g, psi, mb)
    dt = O.dt(g, Rates(), st, u)
    with mmod.Simulation(g, r, "fp32") as sim:
        sim.set_state(psi, mb)
        sim.set_velocity(u)
        sim.set_dt(dt)
        sim.step(3)
        got = sim.get_state()
    O.run(g, r, st, u, dt, 3)
    for k in ("psi", "mb", "c"):
        assert rel_l2(got[k], getattr(st, k)) <= 1e-5, k


def test_batch_groups(mmod):
    """A batch whose members are too many for one group (their Mb together is
    above a group's share of the L2) with one that no resident launch holds:
    every member equals itself stepped alone by single substeps."""
    grids = [Grid(96, 96, 32, 32), Grid(16, 16, 16, 16), Grid(80, 72, 32, 32), Grid(33, 20, 8, 12),
             Grid(128, 128, 32, 32), Grid(64, 48, 16, 20), Grid(96, 64, 64, 64), Grid(192, 128, 64, 48)]
    rates = [Rates(k_off=0.3 + 0.2 * i, glide=0.2) for i in range(len(grids))]
    states = [inputs(g, 20 + i, 0.3) for i, g in enumerate(grids)]
    with mmod.Batch(grids, rates, "fp32") as b:
        for sim, (psi, mb, u) in zip(b.members, states):
            sim.set_state(psi, mb)
            sim.set_velocity(u)
        b.step(3)
        b.members[2].step(2)  # one member alone in between
        b.step(2)
        b.sync()
        got = [sim.get_state() for sim in b.members]
    for i, (g, r, (psi, mb, u)) in enumerate(zip(grids, rates, states)):
        with mmod.Simulation(g, r, "fp32") as sim:
            sim.set_state(psi, mb)
            sim.set_velocity(u)
            for _ in range(7 if i == 2 else 5):
                sim.step(1)
            ref = sim.get_state()
        for k in KEYS:
            assert rel_l2(got[i][k], ref[k]) <= 1e-6, (i, k)


@pytest.mark.parametrize("dims,handles", [((16, 16, 16, 16), 12), ((32, 32, 16, 16), 6),
                                          ((20, 17, 24, 30), 5), ((48, 40, 8, 12), 4)])
def test_small_instances_side_by_side(mmod, dims, handles):
    """Handles on a stream each, their launches on the chip together, with a large one
    that takes all of it among them, calls of many substeps and of few: every result
    is that of the handle alone, bit for bit."""
    import torch
    grids = [Grid(*dims)] * handles + [Grid(96, 80, 32, 32)]
    streams = [torch.cuda.Stream() for _ in grids]
    got = []
    for together in (False, True):
        sims = []
        for i, (g, s) in enumerate(zip(grids, streams)):
            sim = mmod.Simulation(g, Rates(k_off=0.5 + 0.1 * i), "fp32", stream=s.cuda_stream)
            psi, mb, u = inputs(g, 3 + i, 0.3)
            sim.set_state(psi, mb)
            sim.set_velocity(u)
            sims.append(sim)
        calls = (40, 33, 5, 64)
        order = ([(i, n) for n in calls for i in range(len(sims))] if together
                 else [(i, n) for i in range(len(sims)) for n in calls])
        for i, n in order:
            sims[i].step(n)
            if not together:
                sims[i].sync()
        got.append([sim.get_state() for sim in sims])
        for sim in sims:
            sim.close()
    for i, (a, b) in enumerate(zip(*got)):
        for k in KEYS:
            assert np.array_equal(a[k], b[k]), (i, k)


def test_autotune_times_the_tiles_in_use(mmod):
    """A batch with a member that goes over tiles beside one that does not: the tuned
    plan, and the launch information, are those of the first one's tiles."""
    grids = [Grid(64, 64, 32, 32), Grid(192, 128, 64, 48)]
    with mmod.Batch(grids, [Rates()] * 2, "fp32") as b:
        for i, sim in enumerate(b.members):
            psi, mb, u = inputs(sim.grid, 7 + i, 0.3)
            sim.set_state(psi, mb)
            sim.set_velocity(u)
        before = [sim.get_state() for sim in b.members]
        res = b.autotune(substeps=1)
        info = b.launch_info()
        after = [sim.get_state() for sim in b.members]
        b.step(3)
        b.sync()
    assert len(res) == 36
    for x, y in zip(before, after):
        for k in KEYS:
            assert np.array_equal(x[k], y[k]), k
    cells = max(1, info["tile_work"] // (64 * 48))  # of a tile
    assert info["tiles"] == -(-192 * 128 // cells)
