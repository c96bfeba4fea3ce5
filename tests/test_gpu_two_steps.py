"""Two FP32 steps in one launch against the one-step kernels.

Both run the same operations on every node, so at tau = 1 the states agree bit
for bit: at the smallest lattices, at one tile and its edges (62 columns, 6 or 8
rows), at odd sizes, with both launch shapes (the last two sizes take the large one), on walled, periodic and mixed sides, with a porosity field
and an acceleration profile, for even and odd step counts.  Off tau = 1 the
wall nodes' products may contract differently: FP32 rounding (1e-6 after 6
steps, as for the other kernels)."""
import numpy as np
import pytest

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu

D, A, P = "dirichlet", "adiabatic", "periodic"
SIDES = {
    "cavity": dict(bc=(D, D, A, A)),
    "mixed": dict(bc=(D, A, D, A), T_bc=(1.0, 0.0, 0.8, 0.0), u_bc=((0.0, 0.0), (0.0, 0.0), (0.0, 0.0), (0.01, 0.0))),
    "channel": dict(bc=(P, P, D, D), T_bc=(0.0, 0.0, 0.2, 0.9), u_bc=((0.0, 0.0), (0.0, 0.0), (0.0, 1e-3), (0.01, 1e-3))),
    "shaft": dict(bc=(A, D, P, P), T_bc=(0.0, 0.3, 0.0, 0.0)),
    "box": dict(bc=(P, P, P, P)),
}
SIZES = [(8, 8), (9, 11), (62, 18), (63, 19), (64, 20), (125, 37), (131, 8), (300, 130), (1301, 203), (1302, 201)]


def _run(p, fields, steps, two, eps=None, ay=None):
    g = lbm.Lattice(p, "f32")
    g.set_fields(*fields, eps_field=eps)
    if ay is not None:
        g.set_force_profile(ay)
    if not two:
        g.staged = False
    before = g.launches
    g.step(steps)
    g.sync()
    g.check_guards()
    assert g.launches - before == (steps // 2 + steps % 2 if two else steps)
    f, h = g.get_state()
    return f[1:], h


@pytest.mark.parametrize("sides", sorted(SIDES))
@pytest.mark.parametrize("nx,ny", SIZES)
def test_two_steps_match_the_global_load_kernel(nx, ny, sides):
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, Q=1e-5, ax=1e-6, **SIDES[sides])
    fields = W.random_fields(p, seed=nx + ny, amp_u=2e-3, amp_T=0.3)
    ay = 1e-6 * np.arange(ny)
    for steps in (2, 9):
        a, b = _run(p, fields, steps, True, ay=ay), _run(p, fields, steps, False, ay=ay)
        assert np.all(np.isfinite(b[1]))
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("nx,ny", [(63, 19), (260, 133)])
@pytest.mark.parametrize("sides", ["cavity", "channel"])
def test_two_steps_with_a_porosity_field(nx, ny, sides):
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, **SIDES[sides])
    eps = W.gaussian_random_field(nx, corr=8.0, seed=9)[:ny]
    fields = W.random_fields(p, seed=4, amp_u=2e-3, amp_T=0.3)
    a, b = _run(p, fields, 20, True, eps), _run(p, fields, 20, False, eps)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("sides", sorted(SIDES))
def test_two_steps_off_tau_one(sides):
    p = W.cavity(130, 1e5, 1e-3, 0.45, ny=41, tau_f=0.8, tau_T=1.15, Q=1e-4, ax=1e-7, **SIDES[sides])
    fields = W.random_fields(p, seed=8, amp_u=2e-3, amp_T=0.3)
    a, b = _run(p, fields, 6, True), _run(p, fields, 6, False)
    assert np.abs(a[0] - b[0]).max() <= 1e-6 * np.abs(b[0]).max()
    assert np.abs(a[1] - b[1]).max() <= 1e-6 * np.abs(b[1]).max()


def test_a_non_finite_value_is_reported():
    p = W.cavity(70, 1e5, 1e-3, 0.5, ny=40)
    T, ux, uy = W.random_fields(p, seed=1)
    g = lbm.Lattice(p, "f32")
    g.set_fields(T, ux, uy)
    f, h = g.get_state()
    f[0] = 0.0
    h[3, 20, 30] = np.inf
    g.set_state(f, h)
    g.step(2)
    with pytest.raises(lbm.LbmError) as e:
        g.sync()
    assert e.value.status == -3
