"""The float32 substep sums n_b over a row in one order, whatever kernel takes
the row: V nodes to a lane (V the widest of 8, 4 and 1 that divides ns), a lane's
even and odd nodes apart, then the lanes in halving strides. Gradients depend on
it: the Superbee branches of nearly tied differences follow the last bits."""
import numpy as np
import pytest

from paper_1908_04279_gb300.inputs import Grid, Rates, SplitMix64, psi_isotropic_perturbed, random_divfree_flow

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


def row_sums(m):
    """The rows' sums (last axis) in float32, in the order above."""
    ns = m.shape[-1]
    V = 8 if ns % 8 == 0 else 4 if ns % 4 == 0 else 1
    lanes = m.astype(np.float32).reshape(*m.shape[:-1], ns // V, V)
    if V == 1:
        s = lanes[..., 0]
    else:
        even, odd = lanes[..., 0], lanes[..., 1]
        for h in range(1, V // 2):
            even, odd = even + lanes[..., 2 * h], odd + lanes[..., 2 * h + 1]
        s = even + odd
    n = 1
    while n < s.shape[-1]:
        n *= 2
    s = np.concatenate([s, np.zeros((*s.shape[:-1], n - s.shape[-1]), np.float32)], -1)
    while n > 1:
        n //= 2
        s = s[..., :n] + s[..., n:2 * n]
    return s[..., 0]


# rows of one lane and of several, full and not, of an even, an odd and a fourth
# number of nodes, with and without a power of two of lanes; one substep per
# call (the streaming kernel) and three (the resident one)
@pytest.mark.parametrize("ns", [3, 7, 8, 10, 12, 13, 16, 18, 20, 23, 24, 27, 28, 30, 31, 32, 36,
                                44, 52, 60, 64])
@pytest.mark.parametrize("nth", [8, 37])
@pytest.mark.parametrize("n", [1, 3])
def test_row_sum_order(mmod, nth, ns, n):
    """One filament orientation per cell, at rest, and nodes one apart: the coarse
    density is that row's n_b times dtheta, one rounding."""
    g = Grid(16, 12, nth, ns, L=float(ns))
    rng = SplitMix64(17 + ns)
    mb = rng.uniforms(g.micro_cells).reshape(g.ny, g.nx, nth, ns).astype(np.float32).astype(float)
    at = (np.arange(g.ncells) % nth).reshape(g.ny, g.nx, 1)
    psi = np.zeros((g.ny, g.nx, nth))
    np.put_along_axis(psi, at, 1.0, -1)
    with mmod.Simulation(g, Rates(glide=0.0, k_on=1e-4), "fp32") as sim:
        sim.set_state(psi, mb, np.full((g.ny, g.nx), 1e4))
        sim.set_velocity(np.zeros((2, g.ny, g.nx)))
        sim.set_dt(0.3)
        sim.step(n)
        got = sim.get_state()
    assert np.array_equal(got["psi"], psi)
    nb = np.take_along_axis(row_sums(got["mb"]), at, -1)[..., 0]
    dth = np.float32(2.0 * np.pi / nth)
    assert np.array_equal(got["c"].astype(np.float32), nb * dth)


# the rates' gradients of the polar order in float32, whose forward summed these
# rows one node to a lane; held to 2e-5 of them, the bound of a float32 output
# (their conditioning: another order of the same sums moves them by 2e-4)
@pytest.mark.parametrize("dims,n,want", [
    ((24, 77, 24, 29), 100, (-6.93859910233e-07, -1.46884713887e-06, 2.72361848623e-06)),
    ((70, 69, 11, 23), 90, (-2.4954298426e-05, -6.18057547047e-05, 8.46506490761e-05))])
def test_rate_gradients_of_ragged_rows(mmod, dims, n, want):
    import torch
    from paper_1908_04279_gb300.autograd import micro_steps
    g, r = Grid(*dims), Rates()
    psi = torch.tensor(psi_isotropic_perturbed(g, 5), device="cuda")
    u = torch.tensor(random_divfree_flow(g, 6, 8, 0.1), device="cuda")
    rates = [torch.tensor(x, dtype=torch.float64, requires_grad=True)
             for x in (r.k_off, r.v_walk, r.k_on)]
    with mmod.Simulation(g, r, "fp32") as sim:
        value = micro_steps(sim, psi, u, *rates, n_substeps=n, K=10)
        got = torch.autograd.grad(value, rates)
    for a, b in zip(got, want):
        assert abs(float(a) - b) <= 2e-5 * abs(b), (float(a), b)
