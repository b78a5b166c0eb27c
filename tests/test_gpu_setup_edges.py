"""Edges of the state set-up and the diffusion kernels against the oracle:
line lengths around the segments of the cyclic solve and beyond what shared
memory holds (float64, 1e-12), and motor densities whose row sums leave
float32 (float32, 1e-5)."""
import numpy as np
import pytest

from paper_1908_04279_gb300.inputs import Grid, Rates, SplitMix64, psi_isotropic_perturbed

pytestmark = pytest.mark.gpu


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


# two points; one segment, a segment and a point more, 16 segments and one
# over; a short last segment; more than 32 lines; a line of 900 points (the
# thread-per-line solve); a stiff and a nearly vanishing step
@pytest.mark.parametrize("dims,D,dt", [
    ((2, 3, 4), 0.3, 1.0), ((15, 16, 8), 0.02, 1.0), ((17, 9, 31), 0.01, 1.0),
    ((129, 5, 3), 0.002, 1.0), ((131, 7, 12), 1e-3, 0.3), ((900, 2, 4), 1e-5, 1.0),
    ((20, 24, 16), 40.0, 1.0), ((20, 24, 16), 1e-7, 1e-3)])
def test_cyclic_diffusion(mmod, dims, D, dt):
    from oracle import oracle as O
    g = Grid(*dims, 4)
    psi = psi_isotropic_perturbed(g, 5, amp=0.5)
    with mmod.Simulation(g, Rates(), "fp64") as sim:
        sim.set_state(psi)
        sim.diffuse(D, 0.7 * D, dt)
        got = sim.get_state()["psi"]
    assert rel_l2(got, O.diffuse(g, psi, D, 0.7 * D, dt)) <= 1e-12


@pytest.mark.parametrize("ns", [8, 7])
def test_set_up_beyond_float32_sums(mmod, ns):
    """Row sums and coarse densities above the float32 range (each motor value
    is within it): the scale-down brings the state back."""
    from oracle import oracle as O
    g = Grid(5, 4, 12, ns)
    rng = SplitMix64(3)
    psi = psi_isotropic_perturbed(g, 2)
    mb = 2e38 * (0.5 + 0.5 * rng.uniforms(g.micro_cells).reshape(g.ny, g.nx, g.ntheta, g.ns))
    mb[1:] = 0.2  # and cells that are not scaled
    st = O.make_state(g, psi, mb)
    with mmod.Simulation(g, Rates(), "fp32") as sim:
        sim.set_state(psi, mb)
        got = sim.get_state()
    for k in ("mb", "c"):
        assert rel_l2(got[k], getattr(st, k)) <= 1e-5, k
    assert np.abs(got["mf"] - st.mf).max() <= 1e-6


def _walk(M, v_ds):
    """-dPhi/ds of the Superbee-limited walking flux, signs compared instead of
    multiplied (the oracle's products of differences underflow below 1e-160)."""
    def minmod(x, y):
        return np.where(np.sign(x) == np.sign(y), np.sign(x) * np.minimum(abs(x), abs(y)), 0.0)
    a = np.diff(M, axis=-1, prepend=0.0)[..., :-1]
    b = np.diff(M, axis=-1)
    x, y = minmod(2 * a, b), minmod(a, 2 * b)
    slope = np.where(abs(x) > abs(y), x, y)
    F = M.copy()
    F[..., :-1] += 0.5 * slope
    return -v_ds * np.diff(F, axis=-1, prepend=0.0)


@pytest.mark.parametrize("dims", [(7, 6, 12, 16), (6, 5, 10, 13)])
def test_subnormal_motor_densities(mmod, dims):
    """The float64 limiter halves differences on their bit patterns: motor
    densities from zero through the subnormal range (no binding) against the
    scheme in numpy."""
    g = Grid(*dims)
    r = Rates(k_on=0.0)
    rng = SplitMix64(9)
    x = rng.uniforms(2 * g.micro_cells).reshape(2, g.ny, g.nx, g.ntheta, g.ns)
    mb = np.where(x[1] < 0.2, 0.0, 8e-308 * x[0] ** 3)
    psi = psi_isotropic_perturbed(g, 4)
    u = np.zeros((2, g.ny, g.nx))
    dt = 0.4 / g.ns
    with mmod.Simulation(g, r, "fp64") as sim:
        sim.set_state(psi, mb)
        sim.set_velocity(u)
        sim.set_dt(dt)
        sim.step(3)
        got = sim.get_state()
    v_ds = r.v_walk * g.ns
    for _ in range(3):
        half = mb + 0.5 * dt * (_walk(mb, v_ds) - r.k_off * mb)
        mb = mb + dt * (_walk(half, v_ds) - r.k_off * half)
    scale = 1e308  # out of the subnormal range for the norms
    assert rel_l2(got["mb"] * scale, mb * scale) <= 1e-12
    assert rel_l2(got["psi"], psi) <= 1e-12


# the float32 tangent at each width of a lane (eight nodes: 32, 64, 56 to a row,
# 7 of 8 lanes a row; four: an odd cell of few passes; two; one), with more and
# fewer than 32 orientations, against float64 from the same float32 inputs:
# three substeps of some twenty roundings of 2^-24, differences of neighbouring
# nodes losing up to a factor 5
@pytest.mark.parametrize("dims", [(6, 5, 32, 32), (5, 4, 40, 64), (4, 3, 10, 56), (7, 4, 33, 24),
                                  (5, 3, 16, 8), (5, 4, 7, 6), (3, 4, 35, 5)])
def test_tangent_widths(mmod, dims):
    g = Grid(*dims)
    rng = SplitMix64(11)
    psi = psi_isotropic_perturbed(g, 12, amp=0.3).astype(np.float32).astype(np.float64)
    mb = (0.3 * rng.uniforms(g.micro_cells)).reshape(g.ny, g.nx, g.ntheta, g.ns)
    mb = mb.astype(np.float32).astype(np.float64)
    u = 0.2 * (rng.uniforms(2 * g.ny * g.nx).reshape(2, g.ny, g.nx) - 0.5)
    u = u.astype(np.float32).astype(np.float64)
    got = {}
    for precision in ("fp64", "fp32"):
        with mmod.Simulation(g, Rates(v_sp=0.1, glide=0.5, k_on=1.3, k_off=0.7), precision) as sim:
            sim.set_tangent((1.0, 0.3, -0.5))
            sim.set_state(psi, mb, np.full((g.ny, g.nx), 4.0))
            sim.set_velocity(u)
            sim.set_dt(0.004)
            sim.step(3)
            got[precision] = {**sim.get_tangent(), **{"s_" + k: sim.get_state()[k]
                                                      for k in ("psi", "mb", "mf")}}
    for k, v in got["fp64"].items():
        assert rel_l2(got["fp32"][k], v) <= 2e-5, k


@pytest.mark.parametrize("nth,ns", [(8, 6), (40, 32), (5, 30)])
def test_free_motors_of_a_float32_state_under_cancellation(mmod, nth, ns):
    """Mf = M - C of a loaded float32 state is formed in float64: with one motor
    value and one filament density per cell C is a product of four factors (four
    roundings of 2^-53), M the next float32 above it, and Mf is rounded once."""
    g = Grid(64, 48, nth, ns)
    rng = SplitMix64(83)
    k, j = ((rng.uniforms(g.ncells) * n).astype(int) for n in (nth, ns))
    p, m = ((0.2 + rng.uniforms(g.ncells)).astype(np.float32).astype(float) for _ in range(2))
    psi, mb = np.zeros((g.ncells, nth)), np.zeros((g.ncells, nth, ns))
    at = np.arange(g.ncells)
    psi[at, k], mb[at, k, j] = p, m
    C = p.astype(np.longdouble) * m * (g.L / ns) * (2 * np.pi / nth)
    M = np.nextafter(C.astype(np.float32), np.float32(np.inf)).astype(float)
    with mmod.Simulation(g, Rates(), "fp32") as sim:
        sim.set_state(psi.reshape(g.ny, g.nx, -1), mb.reshape(g.ny, g.nx, nth, ns),
                      M.reshape(g.ny, g.nx))
        got = sim.get_state()["mf"].reshape(-1)
    want = M - C
    off = np.abs(got - want) - 2.0 ** -24 * np.abs(want) - 4 * 2.0 ** -53 * C
    assert np.all(off <= 0), float(np.max(off / C) * 2.0 ** 53)
