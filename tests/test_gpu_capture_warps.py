"""The capture-radius motor kernel with one warp to an anchor (more anchors than
blocks, few chunks of configurations) and with four, free and with the scale-down
at the anchors, against the oracle (relative 1e-12 in float64)."""
import pytest

from paper_1908_04279_gb300.inputs import Grid, Rates
from tests.test_gpu_capture import _gpu_run, _inputs, mmod, rel  # noqa: F401

pytestmark = pytest.mark.gpu


def chunks(lines, most=256):
    """Consecutive whole lines, at most `most` configurations a chunk."""
    n, room = 0, 0
    for length in lines[:, 4]:
        if length > room:
            n, room = n + 1, most
        room -= length
    return n


@pytest.mark.parametrize("dims,want", [
    ((7, 6, 2, 10), 1), ((7, 6, 8, 10), 3), ((7, 6, 20, 10), 8), ((7, 6, 32, 10), 12),
    ((33, 29, 4, 6), 1), ((31, 30, 8, 6), 2), ((33, 29, 16, 10), 6), ((34, 30, 32, 10), 12)])
@pytest.mark.parametrize("clip", [False, True])
def test_warps_of_an_anchor(mmod, oracle_mod, dims, want, clip):  # noqa: F811
    O = oracle_mod
    g, rc = Grid(*dims), 1.2 / dims[0]
    r = Rates(ell=2.3 / dims[0], k_on=60.0 if clip else 1.6, glide=0.2)
    more = dict(mb_scale=0.05, mtot_lo=0.02, mtot_span=0.03) if clip else {}
    tpl, psi, mb, mtot, u = _inputs(O, g, r, rc, 431, **more)
    assert chunks(tpl.lines) == want
    st = O.make_state_rc(g, r, rc, psi, mb, mtot)
    dt = (4.0 if clip else 0.7) * O.dt(g, r, O.make_state(g, psi), u)
    clipped = False
    got, _, _ = _gpu_run(mmod, g, r, rc, "fp64", psi, mb, mtot, u, dt, 4)
    for _ in range(4):
        O.run_rc(g, r, rc, st, u, dt, 1)
        clipped = clipped or st.mf.min() == 0.0
    assert clipped == clip
    for k in ("psi", "mb", "mf", "c"):
        assert rel(got[k], getattr(st, k)) <= 1e-12, (k, rel(got[k], getattr(st, k)))
