"""The streaming kernels over row plans with a short last chunk and in either form
of the rows (packed, or a few nodes to a lane), against the oracle: relative L2
1e-12 in float64 and 1e-5 in float32 (single substeps: the streaming kernel)."""
import numpy as np
import pytest

from paper_1908_04279_gb300.inputs import Grid, Rates, SplitMix64, psi_isotropic_perturbed, random_divfree_flow

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5}


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
    return np.linalg.norm(np.asarray(a, dtype=np.float64) - b) / np.linalg.norm(b)


def inputs(g, seed):
    rng = SplitMix64(seed)
    mb = 0.3 * rng.uniforms(g.micro_cells).reshape(g.ny, g.nx, g.ntheta, g.ns)
    return psi_isotropic_perturbed(g, seed, amp=0.3), mb, random_divfree_flow(g, seed + 1, 5, 0.15)


def oracle_run(g, r, seed, n):
    from oracle import oracle as O
    psi, mb, u = inputs(g, seed)
    st = O.make_state(g, psi, mb)
    dt = O.dt(g, r, st, u)
    O.run(g, r, st, u, dt, n)
    return dt, st


SHAPES = [("fp64", 31, 32), ("fp64", 37, 31), ("fp64", 8, 8), ("fp64", 8, 7), ("fp64", 20, 32),
          ("fp64", 46, 48), ("fp64", 62, 15), ("fp64", 40, 64), ("fp64", 37, 44),
          ("fp64", 3, 1), ("fp32", 37, 30), ("fp32", 41, 31), ("fp32", 37, 36), ("fp32", 8, 12),
          ("fp32", 40, 28), ("fp32", 62, 60), ("fp32", 37, 32), ("fp32", 31, 20), ("fp32", 34, 6)]


@pytest.mark.parametrize("precision,nth,ns", SHAPES)
def test_streaming_substeps(mmod, precision, nth, ns):
    g = Grid(13, 9, nth, ns)
    r = Rates(glide=0.3, v_sp=0.05)
    psi, mb, u = inputs(g, 5)
    dt, st = oracle_run(g, r, 5, 4)
    with mmod.Simulation(g, r, precision) as sim:
        info = sim.launch_info()
        sim.set_state(psi, mb)
        sim.set_velocity(u)
        sim.set_dt(dt)
        for _ in range(4):
            sim.step(1)
        got = sim.get_state()
    # whole passes of at least four rows where a cell has them
    assert info["chunk_rows"] == nth or info["chunk_rows"] >= 4
    for k in ("psi", "mb", "mf", "c"):
        assert rel_l2(got[k], getattr(st, k)) <= TOL[precision], k


# float64 batches whose cheaper form is either, units of one cell and of two, short
# last chunks; float32 members stepped one substep at a time
@pytest.mark.parametrize("precision,dims", [
    ("fp64", [(12, 9, 31, 32), (10, 8, 46, 48)]), ("fp64", [(12, 9, 8, 8), (10, 8, 8, 8)]),
    ("fp64", [(8, 6, 16, 16), (7, 5, 20, 28)]), ("fp32", [(12, 9, 37, 28), (10, 8, 16, 16)]),
    ("fp32", [(8, 6, 37, 32), (8, 6, 8, 24)])])
def test_batch_tiles(mmod, precision, dims):
    grids = [Grid(*d) for d in dims]
    r = Rates(glide=0.3)
    with mmod.Batch(grids, [r] * len(grids), precision) as b:
        for i, (g, sim) in enumerate(zip(grids, b.members)):
            psi, mb, u = inputs(g, 7 + i)
            sim.set_state(psi, mb)
            sim.set_velocity(u)
            sim.set_dt(oracle_run(g, r, 7 + i, 0)[0])
        for _ in range(3):
            b.step(1)
        b.sync()
        got = [sim.get_state() for sim in b.members]
    for i, g in enumerate(grids):
        _, st = oracle_run(g, r, 7 + i, 3)
        for k in ("psi", "mb", "mf", "c"):
            assert rel_l2(got[i][k], getattr(st, k)) <= TOL[precision], (i, k)


def test_fp64_batch_equals_alone_in_either_form(mmod):
    """The members of a float64 batch share one form of the rows, which need not be the
    form of a member alone: the same bits all the same."""
    for dims in ([(12, 9, 8, 8), (20, 16, 31, 32)], [(40, 30, 8, 8), (6, 4, 20, 28)],
                 [(9, 7, 8, 12), (24, 20, 34, 30)]):
        grids = [Grid(*d) for d in dims]
        r = Rates(glide=0.3)
        with mmod.Batch(grids, [r] * 2, "fp64") as b:
            for i, sim in enumerate(b.members):
                psi, mb, u = inputs(sim.grid, 7 + i)
                sim.set_state(psi, mb)
                sim.set_velocity(u)
            b.step(5)
            b.sync()
            got = [sim.get_state() for sim in b.members]
        for i, g in enumerate(grids):
            psi, mb, u = inputs(g, 7 + i)
            with mmod.Simulation(g, r, "fp64") as sim:
                sim.set_state(psi, mb)
                sim.set_velocity(u)
                sim.step(5)
                ref = sim.get_state()
            for k in ("psi", "mb", "mf", "c"):
                assert np.array_equal(got[i][k], ref[k]), (dims, i, k)
