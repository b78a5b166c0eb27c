"""Workloads of the microscale kinetic step, as programs that use it run them.

A case names a kind of call, a grid (nx x ny cells, ntheta orientations, ns
arclength nodes), a precision ("fp32" is the mixed form) and the substeps n of
one pass. Arrays live in float64 CUDA tensors, as the library takes and gives
them; a program on the mixed form keeps what it reads back in float32, the
precision of that state, so its outputs here are float32 copies.

Kinds, each one pass through the public entry points:
  forward  a macro step under a prescribed flow: set_velocity, n substeps,
           moments, the state read back. start: "isotropic" begins each pass
           from a perturbed isotropic psi with no motors bound, "saved" from a
           state saved mid-run, "running" goes on from the pass before
  ensemble n substeps of a batch of uneven members, their states read back
  adjoint  torch.autograd: forward of n substeps, polar order, backward
  tangent  n substeps with the tangent along (k_off, v_walk, k_on)
  anchors  a running macro step with the motors anchored under their heads
  capture  a running macro step with a finite capture radius
  local    motor kinetics over a macro interval with a local substep per cell
  alg1     the closed macro loop: fluid solve, n substeps, diffusion, moments
"""
import math

import numpy as np
import torch

from paper_1908_04279_gb300 import mm
from paper_1908_04279_gb300.autograd import micro_steps
from paper_1908_04279_gb300.inputs import Grid, Rates

ELL = 0.05                       # l/L of the kinds with anchors
EPS, Z0 = 0.1, 0.1               # thin-gap fluid solve
D_T, D_R = 1e-3, 0.1             # diffusivities of the macro loop
TANGENT = (1.0, 0.3, 0.0)        # direction of the rates (k_off, v_walk, k_on)
CHECKPOINT = 10                  # adjoint checkpoint interval
MOST_UPDATES = 5.0e10            # motor updates of the largest pass


def _case(kind, nx, ny, ntheta, ns, n, prec="fp32", **more):
    return dict(kind=kind, nx=nx, ny=ny, ntheta=ntheta, ns=ns, n=n, prec=prec, **more)


def listed():
    return [
        # one small run from its initial data, the size of a parameter scan's
        # members and of the cellular-flow workload: launches and latency
        dict(_case("forward", 32, 32, 16, 16, 200, start="isotropic"), name="small_run"),
        # the ordinary macro step of a running simulation (its motors about
        # half of the L2)
        dict(_case("forward", 128, 128, 32, 32, 50, start="running"), name="macro_128"),
        # the largest macro step, far beyond the L2
        dict(_case("forward", 512, 512, 64, 64, 40, start="running"), name="macro_512"),
        # the float64 form, restarted from a saved state
        dict(_case("forward", 128, 128, 32, 32, 20, "fp64", start="saved"), name="macro_fp64"),
        # sizes a resolution study passes through: a grid of odd sides, rows
        # that are not a whole number of vectors
        dict(_case("forward", 85, 61, 24, 30, 50, start="saved"), name="ragged"),
        # a detachment-rate sweep as a batch of uneven instances
        dict(_case("ensemble", 128, 128, 32, 32, 100, members=12), name="ensemble"),
        # inverse problems: the gradient of the polar order
        dict(_case("adjoint", 64, 64, 32, 32, 100), name="adjoint_64"),
        # sensitivity to one direction of the rates in forward mode
        dict(_case("tangent", 128, 128, 32, 32, 50), name="tangent_128"),
        # the non-local motor models
        dict(_case("anchors", 128, 128, 32, 32, 50), name="anchors_128"),
        dict(_case("capture", 64, 64, 32, 32, 30, reach=1.5), name="capture_64"),
        # frozen-psi motor kinetics with independent time steps
        dict(_case("local", 128, 128, 32, 32, 50), name="local_128"),
        # the whole macro loop of the method
        dict(_case("alg1", 128, 128, 32, 32, 50), name="alg1_128"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed kinds: sides and substeps over their ranges, and
    no pass with more motor updates (weighted by what one costs) than the
    largest listed one."""
    kind = rng.choice(["forward"] * 5 + ["ensemble", "adjoint", "tangent", "anchors", "capture",
                                         "local", "alg1"])
    prec = "fp64" if kind in ("forward", "local", "anchors") and rng.random() < 0.2 else "fp32"
    hi = dict(forward=512, ensemble=128, adjoint=96, tangent=256, anchors=256, capture=96,
              local=256, alg1=256)[kind]
    weight = dict(adjoint=8, tangent=4, anchors=4, capture=100, local=2).get(kind, 1)
    if prec == "fp64":
        weight *= 32
    while True:
        c = _case(kind, _log(rng, 24, hi), _log(rng, 24, hi), _log(rng, 8, 64), _log(rng, 8, 64),
                  _log(rng, 20, 200), prec)
        if rng.random() < 0.6:  # round sizes as configurations have them
            for k in ("nx", "ny", "ntheta"):
                c[k] = max(8, c[k] // 8 * 8)
            c["ns"] = rng.choice([16, 32, 64])
        if prec == "fp64":      # a row spans at most one warp
            c["ns"] = c["ns"] // 2 * 2 if c["ns"] > 32 else c["ns"]
        elif c["ns"] > 32 or kind == "ensemble":
            c["ns"] = max(8, c["ns"] // 4 * 4)
        if kind == "capture":
            c["reach"] = rng.choice([1.0, 1.5, 2.0])
            c["n"] = max(10, c["n"] // 5)
            c["ny"] = min(96, max(c["ny"], c["nx"] // 2, 24), 2 * c["nx"])
        if kind == "ensemble":
            c["members"] = rng.randint(6, 16)
        if kind == "adjoint":
            c["n"] = max(20, c["n"] // 10 * 10)
        if kind == "forward":
            c["start"] = rng.choice(["isotropic", "saved", "running"])
        cells = c["nx"] * c["ny"] * c["ntheta"] * c["ns"]
        updates = cells * c["n"] * weight * c.get("members", 1)
        if 1e8 <= updates <= MOST_UPDATES and (kind != "adjoint" or cells <= 1.5e7):
            return c


# ------------------------------------------------------------------ inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _grid(c):
    return Grid(c["nx"], c["ny"], c["ntheta"], c["ns"])


def _rates(c):
    return Rates(ell=ELL) if c["kind"] in ("anchors", "capture") else Rates()


def _members(c, seed):
    """Grids and rates of a detachment-rate sweep: the case's sides are the
    largest member's."""
    rng = np.random.default_rng(c["members"] + 7919 * (c["nx"] + c["ns"]))
    got = []
    for m in range(c["members"]):
        f = (1.0, 0.25, 0.375, 0.5, 0.75)[m % 5]
        g = Grid(max(8, int(c["nx"] * f)), max(8, int(c["ny"] * f)),
                 max(8, c["ntheta"] // (1, 2)[(m // 2) % 2]),
                 max(8, c["ns"] // (1, 2)[(m // 3) % 2] // 4 * 4))
        got.append((g, Rates(v_walk=float(rng.uniform(0.5, 2.0)),
                             k_off=float(np.exp(rng.uniform(math.log(0.05), math.log(5.0))))),
                    seed * 1009 + m))
    return got


def _gen(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed) % (1 << 62))


def _rounded(x, prec):
    """In the mixed form a program's state is float32 already."""
    return x.float().double() if prec == "fp32" else x


def _psi(g, seed, prec, amp=0.05):
    """A perturbed isotropic suspension of total number 1."""
    xi = torch.rand((g.ny, g.nx, g.ntheta), generator=_gen(seed), device=_device(),
                    dtype=torch.float64)
    psi = 1.0 + amp * (2.0 * xi - 1.0)
    psi /= psi.sum() * (2.0 * math.pi / g.ntheta) / (g.nx * g.ny)
    return _rounded(psi, prec)


def _motors(g, r, seed, prec):
    """Bound motors of a run under way: the balance of walking and
    unbinding along each filament, varying between filaments and nodes."""
    gen, dev = _gen(seed + 1), _device()
    s = (torch.arange(g.ns, device=dev, dtype=torch.float64) + 0.5) * (g.L / g.ns)
    ramp = 1.0 - torch.exp(-r.k_off * s / r.v_walk) if r.v_walk > 0 else torch.ones_like(s)
    row = torch.rand((g.ny, g.nx, g.ntheta, 1), generator=gen, device=dev, dtype=torch.float64)
    mb = torch.rand((g.ny, g.nx, g.ntheta, g.ns), generator=gen, device=dev, dtype=torch.float64)
    mb.mul_(0.06).add_(0.97).mul_(row.mul_(0.3).add_(0.85)).mul_(0.6 * r.k_on / r.k_off * ramp)
    return _rounded(mb, prec)


def _flow(g, seed, amp=0.1, modes=8):
    """A divergence-free field of random long-wave stream-function modes."""
    rng, dev = np.random.default_rng(seed + 2), _device()
    x = (torch.arange(g.nx, device=dev, dtype=torch.float64) + 0.5)[None, :] / g.nx
    y = (torch.arange(g.ny, device=dev, dtype=torch.float64) + 0.5)[:, None] / g.ny
    u = torch.zeros((2, g.ny, g.nx), device=dev, dtype=torch.float64)
    for _ in range(modes):
        kx, ky = 0, 0
        while kx == 0 and ky == 0:
            kx, ky = (int(v) for v in rng.integers(-4, 5, 2))
        w = torch.cos(2 * math.pi * (kx * x + ky * y) + rng.uniform(0, 2 * math.pi))
        u[0] += ky * w
        u[1] -= kx * w
    return u * (amp / torch.sqrt(u[0] ** 2 + u[1] ** 2).max())


def _template(g, r, r_c):
    """Walking lines (k, dx, dy, j0, len) of one anchor, in the order of the
    state's entries, and the binding weights [ntheta][ns]."""
    lines, w = [], np.zeros((g.ntheta, g.ns))
    dx, dy = 1.0 / g.nx, 1.0 / g.ny
    for k in range(g.ntheta):
        th = k * (2.0 * math.pi / g.ntheta)
        disp = r.ell * g.L * (2 * np.arange(g.ns) + 1 - g.ns) / (2.0 * g.ns)
        hx, hy = disp * math.cos(th) / dx + 0.5, disp * math.sin(th) / dy + 0.5
        mine = []
        for ey in range(int(math.floor(hy.min() - r_c / dy)) - 1,
                        int(math.floor(hy.max() + r_c / dy)) + 2):
            for ex in range(int(math.floor(hx.min() - r_c / dx)) - 1,
                            int(math.floor(hx.max() + r_c / dx)) + 2):
                px = np.maximum(np.maximum(ex - hx, hx - (ex + 1)), 0.0) * dx
                py = np.maximum(np.maximum(ey - hy, hy - (ey + 1)), 0.0) * dy
                near = np.flatnonzero(px * px + py * py <= r_c * r_c)
                w[k, near] += 1.0
                for run in np.split(near, np.flatnonzero(np.diff(near) != 1) + 1):
                    if run.size:
                        mine.append((k, ex, ey, int(run[0]), int(run.size)))
        lines += sorted(mine, key=lambda q: (q[3], q[2], q[1]))
    return np.array(lines), 1.0 / w


def _capture_motors(g, r, r_c, seed, prec):
    """The motors of _motors per anchor: [ny][nx][entries]."""
    lines, w = _template(g, r, r_c)
    dev = _device()
    j = np.concatenate([np.arange(q[3], q[3] + q[4]) for q in lines])
    wt = np.concatenate([w[q[0], q[3]:q[3] + q[4]] for q in lines])
    s = (j + 0.5) * (g.L / g.ns)
    ramp = torch.tensor(0.6 * wt * (1.0 - np.exp(-r.k_off * s / r.v_walk)) * r.k_on / r.k_off,
                        device=dev)
    mb = torch.rand((g.ny, g.nx, j.size), generator=_gen(seed + 1), device=dev,
                    dtype=torch.float64)
    return _rounded(mb.mul_(0.3).add_(0.85).mul_(ramp), prec)


# ----------------------------------------------------------- prepare and run

def _f64(*shape):
    return torch.empty(shape, device=_device(), dtype=torch.float64)


class _Export:
    """Device buffers a program reads a state and its moments back into."""

    def __init__(self, sim, prec, moments=True, nconf=None):
        g = sim.grid
        last = (nconf,) if nconf else (g.ntheta, g.ns)
        self.sim, self.prec = sim, prec
        self.bufs = dict(psi=_f64(g.ny, g.nx, g.ntheta), mb=_f64(g.ny, g.nx, *last),
                         mf=_f64(g.ny, g.nx), c=_f64(g.ny, g.nx))
        if moments:
            self.bufs["fields"] = _f64(12, g.ny, g.nx)
        self.single = ({k: torch.empty_like(v, dtype=torch.float32)
                        for k, v in self.bufs.items()} if prec == "fp32" else None)

    def __call__(self):
        b = self.bufs
        if "fields" in b:
            self.sim.moments(fields=b["fields"])
        self.sim.get_state_into(b["psi"], b["mb"], b["mf"], b["c"])
        if self.single is None:
            return b
        for k, v in b.items():
            self.single[k].copy_(v)
        return self.single


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "ensemble":
        spec = _members(c, seed)
        batch = mm.Batch([g for g, _, _ in spec], [r for _, r, _ in spec], c["prec"])
        for m, (g, r, s) in zip(batch.members, spec):
            m.set_state(_psi(g, s, c["prec"]), _motors(g, r, s, c["prec"]))
            m.set_velocity(_flow(g, s))
        return dict(case=c, batch=batch,
                    out=[_Export(m, c["prec"], moments=False) for m in batch.members])
    g, r = _grid(c), _rates(c)
    sim = mm.Simulation(g, r, c["prec"])
    st = dict(case=c, sim=sim, psi=_psi(g, seed, c["prec"]), u=_flow(g, seed))
    if kind == "adjoint":
        st["psi"] = st["psi"].float().requires_grad_()
        st["u"] = st["u"].float().requires_grad_()
        st["rates"] = [torch.tensor(x, requires_grad=True) for x in (r.k_off, r.v_walk, r.k_on)]
        return st
    if kind == "capture":
        r_c = c["reach"] / g.nx
        tpl = sim.set_capture(r_c)
        sim.set_state(st["psi"], _capture_motors(g, r, r_c, seed, c["prec"]))
        st["out"] = _Export(sim, c["prec"], nconf=tpl["nconf"])
        return st
    if kind == "tangent":
        sim.set_tangent(TANGENT)
        st["mb"] = _motors(g, r, seed, c["prec"])
        st["mtot"] = torch.ones((g.ny, g.nx), device=_device(), dtype=torch.float64)
        st["out"] = _Export(sim, c["prec"], moments=False)
        st["d"] = dict(dpsi=_f64(g.ny, g.nx, g.ntheta), dmb=_f64(g.ny, g.nx, g.ntheta, g.ns),
                       dmf=_f64(g.ny, g.nx))
        st["d32"] = {k: torch.empty_like(v, dtype=torch.float32) for k, v in st["d"].items()}
        return st
    if c.get("start") == "saved":
        st["mb"] = _motors(g, r, seed, c["prec"])
        st["mtot"] = torch.ones((g.ny, g.nx), device=_device(), dtype=torch.float64)
    elif c.get("start") != "isotropic":
        if kind == "anchors":
            sim.set_anchors(True)
        sim.set_state(st["psi"], _motors(g, r, seed, c["prec"]))
        if kind == "alg1":
            sim.fluid_setup(EPS, Z0)
        if kind == "local":
            # the interval that n global substeps of this flow would cover
            sim.set_velocity(st["u"])
            st["T"] = c["n"] * sim.dt
            st["counts"] = torch.empty((g.ny, g.nx), device=_device(), dtype=torch.int32)
    st["out"] = _Export(sim, c["prec"], moments=kind != "local")
    return st


def run(state):
    c = state["case"]
    kind, n = c["kind"], c["n"]
    if kind == "ensemble":
        state["batch"].step(n)
        return [out() for out in state["out"]]
    sim = state["sim"]
    if kind == "adjoint":
        psi, u, rates = state["psi"], state["u"], state["rates"]
        leaves = [psi, u, *rates]
        value = micro_steps(sim, psi, u, *rates, n_substeps=n, K=CHECKPOINT)
        grads = torch.autograd.grad(value, leaves)
        return dict(value=value.detach().float(), psi=grads[0], u=grads[1],
                    rates=[x for x in grads[2:]])
    if kind == "tangent":
        sim.set_state(state["psi"], state["mb"], state["mtot"])
        sim.set_velocity(state["u"])
        sim.step(n)
        d = state["d"]
        sim._check(sim.lib.mm_get_tangent(sim.h, d["dpsi"].data_ptr(), d["dmb"].data_ptr(),
                                          d["dmf"].data_ptr(), 1))
        value, dvalue = sim.tangent_observable("mean_stress")
        for k, v in d.items():
            state["d32"][k].copy_(v)
        return dict(value=value, dvalue=dvalue, state=state["out"](), tangent=state["d32"])
    if kind == "local":
        sim.motor_local_device(state["T"], state["counts"])
        return dict(state=state["out"](), counts=state["counts"])
    if kind == "alg1":
        sim.fluid_solve(dipole=True, u_out=None)
        sim.step(n)
        sim.diffuse(D_T, D_R, n * sim.dt)
        return state["out"]()
    if c.get("start") == "isotropic":
        sim.set_state(state["psi"])
    elif c.get("start") == "saved":
        sim.set_state(state["psi"], state["mb"], state["mtot"])
    sim.set_velocity(state["u"])
    sim.step(n)
    return state["out"]()


# -------------------------------------------------------------------- work

def _substep_work(cells, nth, ns, t):
    """One substep: Mb, psi and n_b read and written once, the free, coarse
    and total motors and the velocity of every cell; 23 operations per node
    (the two limited stages of a row), about 60 per orientation."""
    return (cells * nth * ns * 2 * t + cells * nth * 4 * t + cells * 6 * t,
            cells * nth * (23 * ns + 60))


def work(case):
    """A pass as the sum of its steps. Each substep reads and writes the state
    once: every step of a run needs the one before on the whole grid."""
    c, kind, n = case, case["kind"], case["n"]
    t = 8 if c["prec"] == "fp64" else 4
    if kind == "ensemble":
        total = [0, 0]
        for g, _, _ in _members(c, 0):
            b, f = _substep_work(g.ncells, g.ntheta, g.ns, t)
            out = g.micro_cells + g.ncells * (g.ntheta + 2)
            total[0] += n * b + out * (t + t)
            total[1] += n * f
        return {"bytes": total[0], "flops": total[1]}
    g = _grid(c)
    cells, rows, micro = g.ncells, g.ncells * g.ntheta, g.micro_cells
    b, f = _substep_work(cells, g.ntheta, g.ns, t)
    export = (micro + rows + 2 * cells) * (t + t) + 12 * cells * (8 + t)
    if kind == "adjoint":
        # a forward, and per substep the state and its adjoint read and the
        # adjoint written (the recomputation is the checkpointing's own)
        back = n * (3 * micro * t + 12 * rows * t)
        return {"bytes": n * b + back + rows * 2 * t + cells * 4 * t, "flops": n * f * 3.5}
    if kind == "tangent":
        return {"bytes": 2 * n * b + 3 * (micro + rows) * (8 + t) + cells * 60,
                "flops": n * f * 2.5}
    if kind == "capture":
        lines, _ = _template(g, _rates(c), c["reach"] / g.nx)
        conf, nl = int(lines[:, 4].sum()), len(lines)
        step = cells * (conf * 2 * t + nl * 2 * t + 5 * g.ntheta * t + 4 * t)
        return {"bytes": n * step + cells * (conf + g.ntheta + 2) * 2 * t + 12 * cells * (8 + t),
                "flops": n * cells * 25 * conf}
    if kind == "local":
        # the motors cross memory once, whatever the substeps
        return {"bytes": micro * 2 * t + rows * 2 * t + (micro + rows + 2 * cells) * 2 * t,
                "flops": n * micro * 23}
    if kind == "anchors":
        b += 2 * cells * 8
    extra = 0
    if kind == "alg1":
        extra = 6 * rows * t + micro * t + 128 * (g.nx // 2 + 1) * g.ny
    if kind == "forward" and c["start"] != "running":
        extra += rows * 8 + (micro * 8 if c["start"] == "saved" else micro * t)
    return {"bytes": n * b + micro * t + export + extra, "flops": n * f}


# ------------------------------------------------- the same in 64 bits (torch)

def _superbee(a, b, grad):
    """Superbee slope of backward and forward differences; with `grad` on the
    branch taken, so that torch differentiates that branch."""
    if not grad:
        aa, ab = a.abs(), b.abs()
        mag = torch.maximum(torch.minimum(2 * aa, ab), torch.minimum(aa, 2 * ab))
        return torch.where((a > 0) == (b > 0), torch.copysign(mag, b), torch.zeros_like(a))
    with torch.no_grad():
        aa, ab = a.detach().abs(), b.detach().abs()
        zero = torch.zeros_like(aa)
        same = ((a > 0) == (b > 0)) & (aa > 0) & (ab > 0)
        t1, t2 = torch.minimum(2 * aa, ab), torch.minimum(aa, 2 * ab)
        first, x1, x2 = t1 > t2, 2 * aa < ab, aa < 2 * ab
        ca = torch.where(same, torch.where(first, 2.0 * x1, 1.0 * x2), zero)
        cb = torch.where(same, torch.where(first, 1.0 * ~x1, 2.0 * ~x2), zero)
    return ca * a + cb * b


def _walk(M, last=None, first=None, grad=False):
    """F_{j-1} - F_j of the limited fluxes over the last axis (whole rows, or
    lines from `first` to `last`, masks of that axis)."""
    zero = torch.zeros_like(M[..., :1])
    left = torch.cat([zero, M[..., :-1]], -1)
    if first is not None:
        left = torch.where(first, torch.zeros_like(left), left)
    right = torch.cat([M[..., 1:], zero], -1)
    slope = _superbee(M - left, right - M, grad)
    if last is None:
        slope = torch.cat([slope[..., :-1], zero], -1)
    else:
        slope = torch.where(last, torch.zeros_like(slope), slope)
    F = M + 0.5 * slope
    Fl = torch.cat([zero, F[..., :-1]], -1)
    if first is not None:
        Fl = torch.where(first, torch.zeros_like(Fl), Fl)
    return Fl - F


def _rk2(M, bind, dt, cw, koff, **more):
    Ms = M + 0.5 * dt * (cw * _walk(M, **more) - koff * M + bind)
    return M + dt * (cw * _walk(Ms, **more) - koff * Ms + bind)


def _roll(x, dy, dx):
    return torch.roll(x, (-dy, -dx), (0, 1))


class _Geometry:
    def __init__(self, g, u):
        dev = u.device
        self.g, self.dth, self.ds = g, 2.0 * math.pi / g.ntheta, g.L / g.ns
        k = torch.arange(g.ntheta, device=dev, dtype=torch.float64)
        self.cos, self.sin = torch.cos(k * self.dth), torch.sin(k * self.dth)
        cf, sf = torch.cos((k + 0.5) * self.dth), torch.sin((k + 0.5) * self.dth)
        self.u = u
        ux, uy = u[0], u[1]
        Gxx, Gyx = ((_roll(q, 0, 1) - _roll(q, 0, -1)) * (0.5 * g.nx) for q in (ux, uy))
        Gxy, Gyy = ((_roll(q, 1, 0) - _roll(q, -1, 0)) * (0.5 * g.ny) for q in (ux, uy))
        e = [q[..., None] for q in (Gxx, Gxy, Gyx, Gyy)]
        self.wp = -sf * (e[0] * cf + e[1] * sf) + cf * (e[2] * cf + e[3] * sf)

    def speed(self, r, nb):
        V = r.v_sp + r.glide * nb
        return self.u[0][..., None] - V * self.cos, self.u[1][..., None] - V * self.sin

    def dt(self, r, psi, nb):
        g = self.g
        ax, ay = self.speed(r, nb)
        adv = float((ax.abs() * g.nx + ay.abs() * g.ny).max())
        rot = float(self.wp.abs().max()) / self.dth
        rho = float((psi.sum(-1) * self.dth).max())
        return r.cfl / max(r.v_walk / self.ds, adv, rot, r.k_off + r.k_on * g.L * rho)

    def transport(self, r, dt, psi, nb):
        g = self.g

        def donor(A, left, right):
            return torch.where(A > 0, A * left, A * right)

        ax, ay = self.speed(r, nb)
        Fe = donor(0.5 * (ax + _roll(ax, 0, 1)), psi, _roll(psi, 0, 1))
        Fn = donor(0.5 * (ay + _roll(ay, 1, 0)), psi, _roll(psi, 1, 0))
        Fp = donor(self.wp, psi, torch.roll(psi, -1, -1))
        return psi - dt * ((Fe - _roll(Fe, 0, -1)) * g.nx + (Fn - _roll(Fn, -1, 0)) * g.ny
                           + (Fp - torch.roll(Fp, 1, -1)) / self.dth)


def _close(psi, mb, mtot, ds, dth):
    """Eq. 5, the scale-down, Eq. 6: mb, mf, c (mb scaled where it applies)."""
    C = (psi * (mb.sum(-1) * ds)).sum(-1) * dth
    if bool((mtot < C).any()):
        f = torch.where(mtot < C, mtot / C, torch.ones_like(C))
        mb = mb * f[..., None, None]
        C = torch.minimum(C, mtot)
    return mb, mtot - C, C


def _substep(geo, r, dt, psi, mb, mf, mtot, grad=False):
    """One substep; large motor densities slab by slab in place."""
    g, ds, dth = geo.g, geo.ds, geo.dth
    cw = r.v_walk / ds
    psi = geo.transport(r, dt, psi, mb.sum(-1) * ds)
    if grad:
        new = _rk2(mb, r.k_on * mf[..., None, None], dt, cw, r.k_off, grad=True)
        C = (psi * (new.sum(-1) * ds)).sum(-1) * dth
        return psi, new, mtot - C, C
    c = torch.empty_like(mf)
    rows = max(1, (1 << 26) // (g.nx * g.ntheta * g.ns))
    for y in range(0, g.ny, rows):
        q = slice(y, y + rows)
        new = _rk2(mb[q], r.k_on * mf[q][..., None, None], dt, cw, r.k_off)
        mb[q], mf[q], c[q] = _close(psi[q], new, mtot[q], ds, dth)
    return psi, mb, mf, c


def _fields(geo, r, psi, mb, mf, c, force=None, rows=None):
    g, dth, ds = geo.g, geo.dth, geo.ds
    ct, st = geo.cos, geo.sin
    s = -0.5 * g.L + (torch.arange(g.ns, device=psi.device, dtype=torch.float64) + 0.5) * ds
    nb, m1 = rows if rows is not None else (mb.sum(-1) * ds, (mb @ s) * ds)
    F, e = r.force_scale, r.force_scale * r.ell
    w = [psi, psi * ct, psi * st, psi * (ct * ct - 0.5), psi * ct * st]
    out = [q.sum(-1) * dth for q in w] + [c, mf]
    out += ([F * (psi * nb * q).sum(-1) * dth for q in (ct, st)] if force is None else list(force))
    out += [e * (psi * m1 * q).sum(-1) * dth for q in (ct * ct, ct * st, st * st)]
    return torch.stack(out)


def _diffuse(g, psi, dt):
    """Crank-Nicolson in each direction, by its Fourier amplification."""
    for axis, n, h, D in ((2, g.ntheta, 2 * math.pi / g.ntheta, D_R), (1, g.nx, 1.0 / g.nx, D_T),
                          (0, g.ny, 1.0 / g.ny, D_T)):
        q = (D * dt / (h * h)) * (1.0 - torch.cos(2 * math.pi * torch.arange(
            n, device=psi.device, dtype=torch.float64) / n))
        amp = ((1.0 - q) / (1.0 + q)).reshape([-1 if a == axis else 1 for a in range(3)])
        psi = torch.fft.ifft(torch.fft.fft(psi, dim=axis) * amp, dim=axis).real
    return psi


def _response(kappa):
    """(g_T, g_L) at wavenumbers kappa > 0: the in-plane velocity at z0 per
    unit force there, across k (a Dirichlet Green's function) and along k (w
    of the thin-gap equations on both sides of the plane from the
    exponentials exp(+-kappa z), exp(+-eps kappa z), with w = w' = 0 on the
    plates, a jump kappa eps^2 of w'' at z0 and w, w', w''' continuous)."""
    mu = EPS * kappa
    gT = EPS ** 2 * (-torch.expm1(-2 * mu * Z0)) * (-torch.expm1(-2 * mu * (1 - Z0))) / (
        2 * mu * (-torch.expm1(-2 * mu)))
    A = torch.zeros((kappa.numel(), 8, 8), device=kappa.device, dtype=torch.float64)
    b = torch.zeros((kappa.numel(), 8, 1), device=kappa.device, dtype=torch.float64)

    def basis(side, z, order):
        lo, hi = (0.0, Z0) if side == 0 else (Z0, 1.0)
        got = []
        for m in (kappa, mu):
            q = m / kappa
            got += [(-q) ** order * torch.exp(-m * (z - lo)), q ** order * torch.exp(m * (z - hi))]
        return torch.stack(got, -1)

    for row, order in ((0, 0), (1, 1)):
        A[:, row, :4] = basis(0, 0.0, order)
        A[:, 2 + row, 4:] = basis(1, 1.0, order)
    for order in range(4):
        A[:, 4 + order, :4] = -basis(0, Z0, order)
        A[:, 4 + order, 4:] = basis(1, Z0, order)
    b[:, 6, 0] = EPS ** 2 / kappa
    x = torch.linalg.solve(A, b)[:, :4, 0]
    return gT, -(basis(0, Z0, 1) * x).sum(-1)


def _fluid(g, F, sigma):
    """u on the filament plane from the force and minus the force dipole."""
    Fh = torch.fft.fft2(F)
    Sh = torch.fft.fft2(-sigma)
    dev = F.device
    total = 0
    for sx in (1.0, -1.0):
        for sy in (1.0, -1.0):  # a Nyquist wavenumber stands for both signs
            k = []
            for n, sg in ((g.nx, sx), (g.ny, sy)):
                m = torch.fft.fftfreq(n, device=dev, dtype=torch.float64) * n
                if n % 2 == 0:
                    m[n // 2] = sg * n / 2
                k.append(2 * math.pi * m)
            kx, ky = k[0][None, :].expand(g.ny, g.nx), k[1][:, None].expand(g.ny, g.nx)
            kap = torch.sqrt(kx * kx + ky * ky)
            uniq, inv = torch.unique(kap[kap > 0], return_inverse=True)
            rT, rL = _response(uniq)
            gT = torch.full_like(kap, EPS ** 2 * Z0 * (1 - Z0))
            gL = gT.clone()
            gT[kap > 0], gL[kap > 0] = rT[inv], rL[inv]
            f = torch.stack([Fh[0] + 1j * (kx * Sh[0] + ky * Sh[1]),
                             Fh[1] + 1j * (kx * Sh[1] + ky * Sh[2])])
            hat = torch.stack([kx, ky]) / torch.where(kap > 0, kap, torch.ones_like(kap))
            total = total + gT * f + (gL - gT) * hat * (hat * f).sum(0)
    return torch.fft.ifft2(total / 4).real.contiguous()


def _heads(g, r):
    """Cell offsets (ox, oy) [ntheta][ns] of the motor heads."""
    disp = r.ell * g.L * (2 * np.arange(g.ns) + 1 - g.ns) / (2.0 * g.ns)
    th = [k * (2.0 * math.pi / g.ntheta) for k in range(g.ntheta)]
    ct, st = np.array([[math.cos(t)] for t in th]), np.array([[math.sin(t)] for t in th])
    return (np.floor(disp * ct / (1.0 / g.nx) + 0.5).astype(int),
            np.floor(disp * st / (1.0 / g.ny) + 0.5).astype(int))


def _shifted(g, ox, oy, dev):
    """Cell index at (x + ox, y + oy) for every cell and offset."""
    x, y = torch.arange(g.nx, device=dev), torch.arange(g.ny, device=dev)
    ox, oy = torch.as_tensor(ox, device=dev), torch.as_tensor(oy, device=dev)
    more = [None] * ox.dim()
    return (((y[(slice(None), None, *more)] + oy) % g.ny) * g.nx
            + (x[(None, slice(None), *more)] + ox) % g.nx)


def _exact_anchors(c, seed):
    g, r = _grid(c), _rates(c)
    psi, mb = _psi(g, seed, c["prec"]), _motors(g, r, seed, c["prec"])
    geo = _Geometry(g, _flow(g, seed))
    at = _shifted(g, *_heads(g, r), psi.device)
    ds, dth, cw = geo.ds, geo.dth, r.v_walk / geo.ds

    def close(psi, mb):
        C = torch.zeros(g.ncells, device=psi.device, dtype=torch.float64)
        C.index_add_(0, at.reshape(-1), (psi[..., None] * mb).reshape(-1) * (ds * dth))
        over = C > 1.0
        if bool(over.any()):
            f = torch.where(over, 1.0 / C, torch.ones_like(C))
            mb, C = mb * f[at], torch.where(over, torch.ones_like(C), C)
        return mb, 1.0 - C, C

    mb, mf, C = close(psi, mb)
    dt = geo.dt(r, psi, mb.sum(-1) * ds)
    for _ in range(c["n"]):
        psi = geo.transport(r, dt, psi, mb.sum(-1) * ds)
        mb, mf, C = close(psi, _rk2(mb, r.k_on * mf[at], dt, cw, r.k_off))
    force = torch.zeros((2, g.ncells), device=psi.device, dtype=torch.float64)
    for q, w in enumerate((geo.cos, geo.sin)):
        force[q].index_add_(0, at.reshape(-1), ((psi * w)[..., None] * mb).reshape(-1)
                            * (r.force_scale * ds * dth))
    mf, C = mf.reshape(g.ny, g.nx), C.reshape(g.ny, g.nx)
    return dict(psi=psi, mb=mb, mf=mf, c=C,
                fields=_fields(geo, r, psi, mb, mf, C, force.reshape(2, g.ny, g.nx)))


def _exact_capture(c, seed):
    g, r = _grid(c), _rates(c)
    r_c = c["reach"] / g.nx
    lines, w = _template(g, r, r_c)
    psi, dev = _psi(g, seed, c["prec"]), _device()
    geo = _Geometry(g, _flow(g, seed))
    ds, dth, cw, nl = geo.ds, geo.dth, r.v_walk / geo.ds, len(lines)
    k = torch.as_tensor(lines[:, 0], device=dev)
    fil = _shifted(g, -lines[:, 1], -lines[:, 2], dev).reshape(g.ncells, nl)  # of each (r0, line)
    row = fil * g.ntheta + k
    j = np.arange(g.ns)[None, :]
    inside = torch.as_tensor((j >= lines[:, 3:4]) & (j < lines[:, 3:4] + lines[:, 4:5]), device=dev)
    first = torch.as_tensor(j == lines[:, 3:4], device=dev)
    last = torch.as_tensor(j == lines[:, 3:4] + lines[:, 4:5] - 1, device=dev)
    wl = torch.as_tensor(w[lines[:, 0]], device=dev) * inside
    M = torch.zeros((g.ncells, nl, g.ns), device=dev, dtype=torch.float64)
    M[:, inside] = _capture_motors(g, r, r_c, seed, c["prec"]).reshape(g.ncells, -1)

    def nb():
        q = torch.zeros(g.ncells * g.ntheta, device=dev, dtype=torch.float64)
        q.index_add_(0, row.reshape(-1), M.sum(-1).reshape(-1) * ds)
        return q.reshape(g.ny, g.nx, g.ntheta)

    def close():
        C = (psi.reshape(-1)[row] * (M.sum(-1) * ds)).sum(-1) * dth
        over = C > 1.0
        if bool(over.any()):
            M.mul_(torch.where(over, 1.0 / C, torch.ones_like(C))[:, None, None])
            C = torch.where(over, torch.ones_like(C), C)
        return 1.0 - C, C

    mf, C = close()
    dt = geo.dt(r, psi, nb())
    step = max(1, (1 << 26) // (nl * g.ns))
    for _ in range(c["n"]):
        psi = geo.transport(r, dt, psi, nb())
        for a in range(0, g.ncells, step):
            q = slice(a, a + step)
            M[q] = _rk2(M[q], r.k_on * mf[q, None, None] * wl, dt, cw, r.k_off, last=last,
                        first=first) * inside
        mf, C = close()
    ox, oy = _heads(g, r)
    force = torch.zeros((2, g.ncells), device=dev, dtype=torch.float64)
    nodes = torch.zeros((g.ncells * g.ntheta, g.ns), device=dev, dtype=torch.float64)
    nodes.index_add_(0, row.reshape(-1), M.reshape(-1, g.ns))
    nodes = nodes.reshape(g.ny, g.nx, g.ntheta, g.ns)
    at = _shifted(g, ox, oy, dev)
    for q, t in enumerate((geo.cos, geo.sin)):
        force[q].index_add_(0, at.reshape(-1), ((psi * t)[..., None] * nodes).reshape(-1)
                            * (r.force_scale * ds * dth))
    mf, C = mf.reshape(g.ny, g.nx), C.reshape(g.ny, g.nx)
    return dict(psi=psi, mb=M[:, inside].reshape(g.ny, g.nx, -1), mf=mf, c=C,
                fields=_fields(geo, r, psi, nodes, mf, C, force.reshape(2, g.ny, g.nx)))


def _start(g, r, psi, mb, geo):
    mtot = torch.ones((g.ny, g.nx), device=psi.device, dtype=torch.float64)
    mb, mf, c = _close(psi, mb, mtot, geo.ds, geo.dth)
    return mb, mf, c, mtot


def _exact_adjoint(c, seed):
    from torch.utils.checkpoint import checkpoint
    g, r = _grid(c), _rates(c)
    psi0 = _psi(g, seed, "fp32").requires_grad_()
    u = _flow(g, seed).float().double().requires_grad_()
    rates = [torch.tensor(x, dtype=torch.float64, device=psi0.device, requires_grad=True)
             for x in (r.k_off, r.v_walk, r.k_on)]

    class R:
        k_off, v_walk, k_on = rates
        glide, v_sp, cfl = r.glide, r.v_sp, r.cfl

    with torch.no_grad():
        none = torch.zeros((g.ny, g.nx, g.ntheta), device=psi0.device, dtype=torch.float64)
        dt = _Geometry(g, u.detach()).dt(r, psi0.detach(), none)
    mtot = torch.ones((g.ny, g.nx), device=psi0.device, dtype=torch.float64)

    def step(psi, mb, mf, u, *_):
        return _substep(_Geometry(g, u), R, dt, psi, mb, mf, mtot, grad=True)[:3]

    state = (psi0, torch.zeros((*psi0.shape, g.ns), device=psi0.device, dtype=torch.float64), mtot)
    for _ in range(c["n"]):
        state = checkpoint(step, *state, u, *rates, use_reentrant=False)
    psi = state[0]
    th = torch.arange(g.ntheta, device=psi0.device, dtype=torch.float64) * (2 * math.pi / g.ntheta)
    sc, ss = (psi * torch.cos(th)).sum(), (psi * torch.sin(th)).sum()
    value = torch.sqrt(sc * sc + ss * ss) / psi.sum()
    grads = torch.autograd.grad(value, [psi0, u, *rates])
    return dict(value=value.detach(), psi=grads[0], u=grads[1], rates=list(grads[2:]))


def _exact_tangent(c, seed):
    from torch.autograd import forward_ad as fw
    g, r = _grid(c), _rates(c)
    psi, mb = _psi(g, seed, c["prec"]), _motors(g, r, seed, c["prec"])
    geo = _Geometry(g, _flow(g, seed))
    mb, mf, C, mtot = _start(g, r, psi, mb, geo)
    dt = geo.dt(r, psi, mb.sum(-1) * geo.ds)
    state, d = (psi, mb, mf), [torch.zeros_like(x) for x in (psi, mb, mf)]
    s = -0.5 * g.L + (torch.arange(g.ns, device=psi.device, dtype=torch.float64) + 0.5) * geo.ds
    for i in range(c["n"] + 1):
        with fw.dual_level():
            dual = [fw.make_dual(x, t) for x, t in zip(state, d)]
            if i == c["n"]:  # mean over cells of tr sigma_a
                v = (dual[0] * (dual[1] @ s)).sum() * (
                    r.force_scale * r.ell * geo.ds * geo.dth / g.ncells)
                value, dvalue = fw.unpack_dual(v)
                break
            rr = [fw.make_dual(torch.tensor(x, dtype=torch.float64, device=psi.device),
                               torch.tensor(t, dtype=torch.float64, device=psi.device))
                  for x, t in zip((r.k_off, r.v_walk, r.k_on), TANGENT)]

            class R:
                k_off, v_walk, k_on = rr
                glide, v_sp = r.glide, r.v_sp

            got = _substep(geo, R, dt, *dual, mtot, grad=True)
            if bool((got[2] < 0).any()):  # a scale-down: not followed here
                return None
            both = [fw.unpack_dual(x) for x in got]
        state, C = tuple(x.primal for x in both[:3]), both[3].primal
        d = [x.tangent for x in both[:3]]
    return dict(value=float(value), dvalue=float(dvalue),
                state=dict(psi=state[0], mb=state[1], mf=state[2], c=C),
                tangent=dict(dpsi=d[0], dmb=d[1], dmf=d[2]))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "anchors":
        return _exact_anchors(c, seed)
    if kind == "capture":
        return _exact_capture(c, seed)
    if kind == "adjoint":
        return _exact_adjoint(c, seed)
    if kind == "tangent":
        return _exact_tangent(c, seed)
    if kind == "ensemble":
        out = []
        for g, r, s in _members(c, seed):
            geo, psi = _Geometry(g, _flow(g, s)), _psi(g, s, c["prec"])
            mb, mf, C, mtot = _start(g, r, psi, _motors(g, r, s, c["prec"]), geo)
            dt = geo.dt(r, psi, mb.sum(-1) * geo.ds)
            for _ in range(c["n"]):
                psi, mb, mf, C = _substep(geo, r, dt, psi, mb, mf, mtot)
            out.append(dict(psi=psi, mb=mb, mf=mf, c=C))
        return out
    g, r, n = _grid(c), _rates(c), c["n"]
    psi, geo = _psi(g, seed, c["prec"]), _Geometry(g, _flow(g, seed))
    if c.get("start") == "isotropic":
        mb = torch.zeros((*psi.shape, g.ns), device=psi.device, dtype=torch.float64)
    else:
        mb = _motors(g, r, seed, c["prec"])
    mb, mf, C, mtot = _start(g, r, psi, mb, geo)
    if kind == "alg1":
        fields = _fields(geo, r, psi, mb, mf, C)
        geo = _Geometry(g, _fluid(g, fields[7:9], fields[9:12]))
    dt = geo.dt(r, psi, mb.sum(-1) * geo.ds)
    if kind == "local":
        rate = torch.clamp(r.k_off + r.k_on * g.L * (psi.sum(-1) * geo.dth), min=r.v_walk / geo.ds)
        counts = torch.clamp(torch.ceil(n * dt * rate / r.cfl), min=1.0)
        own = (n * dt / counts)[..., None, None]
        for i in range(int(counts.max())):
            new = _rk2(mb, r.k_on * mf[..., None, None], own, r.v_walk / geo.ds, r.k_off)
            new, mf1, C1 = _close(psi, new, mtot, geo.ds, geo.dth)
            on = i < counts
            mb = torch.where(on[..., None, None], new, mb)
            mf, C = torch.where(on, mf1, mf), torch.where(on, C1, C)
        return dict(state=dict(psi=psi, mb=mb, mf=mf, c=C), counts=counts.to(torch.int32))
    for _ in range(n):
        psi, mb, mf, C = _substep(geo, r, dt, psi, mb, mf, mtot)
    if kind == "alg1":
        psi = _diffuse(g, psi, n * dt)
        mb, mf, C = _close(psi, mb, mtot, geo.ds, geo.dth)
    return dict(psi=psi, mb=mb, mf=mf, c=C, fields=_fields(geo, r, psi, mb, mf, C))
