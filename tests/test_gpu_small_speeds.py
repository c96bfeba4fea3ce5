"""FP64 lattices whose speeds reach down to where |v|^2 is subnormal or zero
(|v| below 1.5e-154): an eddy with Gaussian tails in fluid at rest, as any localised
disturbance has ahead of its front, against the oracle (1e-10 of the largest
speed, the bound of the FP64 tests), and uniform speeds through that range
one by one.  FP64 keeps subnormal values, so every one of them is met."""
import numpy as np
import pytest

import oracle
from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TINY = np.finfo(np.float64).tiny  # the smallest normal number
REST = dict(T_bc=(0.5, 0.5, 0.5, 0.5))  # every wall at the initial temperature: only the eddy moves


def _eddy(p, width):
    y, x = np.mgrid[0:p["ny"], 0:p["nx"]]
    dx, dy = (x - p["nx"] // 2) / width, (y - p["ny"] // 2) / width
    a = 0.01 * np.exp(-dx * dx - dy * dy)
    return np.full(a.shape, p["T_init"]), a, -0.5 * a


def _met(m):
    """Nodes in the range (the oracle stores g_i whole: its T - T0, and through it u, is rounding noise of 1e-17)."""
    vv = m["ux"] ** 2 + m["uy"] ** 2
    return np.count_nonzero((vv > 0) & (vv < TINY))


def _check(p, fields, steps, eps, m):
    mo = oracle.Oracle(p, *fields, eps_field=eps).run(steps).moments()
    umax = np.sqrt(mo["ux"] ** 2 + mo["uy"] ** 2).max()
    for k in ("ux", "uy"):
        assert np.abs(m[k] - mo[k]).max() <= 1e-10 * umax, k
    assert np.abs(m["T"] - mo["T"]).max() <= 1e-10


# 64 x 48: flow and thermal planes in blocks of their own; 260 x 200: one thread a node
@pytest.mark.parametrize("state", ["populations", "moments"])
@pytest.mark.parametrize("nx,ny,width", [(64, 48, 1.5), (260, 200, 5.0)])
def test_an_eddy_in_fluid_at_rest(nx, ny, width, state):
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, **REST)
    fields = _eddy(p, width)
    g = lbm.Lattice(p, "f64", state=state)
    g.set_fields(*fields)
    assert _met(g.moments()) > 20
    g.step(20)
    assert np.all(np.isfinite(g.residual()))
    g.sync()  # raises if a value is not finite
    _check(p, fields, 20, None, g.moments())


@pytest.mark.parametrize("more", [dict(), dict(tau_f=0.8, tau_T=1.15), dict(bc=("periodic",) * 4)])
def test_an_eddy_in_a_porosity_field(more):
    p = W.cavity(72, 1e5, 1e-3, 0.5, ny=60, **{**REST, **more})
    fields = _eddy(p, 1.5)
    eps = W.gaussian_random_field(72, corr=8.0, seed=3)[:60]
    g = lbm.Lattice(p, "f64")
    g.set_fields(*fields, eps_field=eps)
    assert _met(g.moments()) > 20
    g.step(12)
    g.sync()
    _check(p, fields, 12, eps, g.moments())


def test_eddies_in_a_batch():
    probs = [W.cavity(64, 1e5, 1e-3, 0.5, ny=48, **REST), W.cavity(70, 1e4, 1e-2, 0.7, **REST)]
    b = lbm.Batch(probs, "f64")
    for c, p in enumerate(probs):
        b.set_fields(c, *_eddy(p, 1.5))
        assert _met(b.moments(c)) > 20
    b.step(15)
    b.sync()
    for c, p in enumerate(probs):
        _check(p, _eddy(p, 1.5), 15, None, b.moments(c))


def test_the_gradient_through_an_eddy():
    p = W.cavity(40, 1e4, 1e-2, 0.6, ny=36, **REST)
    T, ux, uy = _eddy(p, 1.0)
    eps = W.gaussian_random_field(40, corr=4.0, seed=4)[:36]
    steps = 30
    g = lbm.Lattice(p, "f64")
    g.set_fields(T, ux, uy, eps_field=eps)
    assert _met(g.moments()) > 5
    loss, g_eps, g_t = g.adjoint(steps)
    o = oracle.Oracle(p, T, ux, uy, eps_field=eps).run(steps)
    assert abs(loss - o.nusselt("W")[0]) <= 1e-10
    # cells where the initial speed is below 1e-20: elsewhere the oracle's derivative also has the initial
    # state's own dependence on the porosity, which the gradient (of a given state) does not
    cells = [(1, 18), (2, 3), (20, 28), (11, 18), (30, 9), (38, 30)]
    assert max(abs(ux[y, x]) for x, y in cells) < 1e-20
    ref, ref_t = oracle.nusselt_gradient(p, steps, eps, cells, sides=("W", "E"), T=T, ux=ux, uy=uy)
    scale = max(np.abs(ref).max(), 1e-12)
    assert np.all(np.isfinite(g_eps))
    for k, (x, y) in enumerate(cells):
        assert g_eps[y, x] == pytest.approx(ref[k], abs=1e-9 * scale), (x, y)
    for s in "WE":
        assert g_t["WESN".index(s)] == pytest.approx(ref_t[s], rel=1e-9, abs=1e-12), s


@pytest.mark.parametrize("state", ["populations", "moments"])
@pytest.mark.parametrize("exponent", range(148, 165, 2))
def test_uniform_speeds_through_the_subnormal_squares(exponent, state):
    p = W.cavity(12, 1e5, 1e-3, 0.5, bc=("periodic",) * 4, gbeta=0.0)
    u = 3.7 * 10.0 ** -exponent
    fields = (np.full((12, 12), 0.5), np.full((12, 12), u), np.full((12, 12), -0.4 * u))
    g = lbm.Lattice(p, "f64", state=state)
    g.set_fields(*fields)
    g.step(3)
    g.sync()
    m, mo = g.moments(), oracle.Oracle(p, *fields).run(3).moments()
    for k in ("ux", "uy"):
        assert np.all(mo[k] != 0.0)
        assert np.abs(m[k] / mo[k] - 1.0).max() <= 1e-12, k
