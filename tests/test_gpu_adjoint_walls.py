"""The reverse-mode adjoint step where its wall handling can go wrong, FP64,
against the oracle's complex-step derivatives (1e-9 of the gradient's scale,
the bound of the adjoint tests): lattices so small that x_f and x_ff of
opposite walls are neighbours or swap places, periodic sides, moving walls,
heat sources and body forces, relaxation times off 1, one block and several."""
import numpy as np
import pytest

import oracle
from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu

D, A, P = "dirichlet", "adiabatic", "periodic"
CASES = [
    (4, 4, dict(bc=(D, D, A, A)), "W"),
    (5, 6, dict(bc=(A, D, A, D), T_bc=(1.0, 0.0, 0.6, 0.3)), "N"),
    (7, 5, dict(bc=(D, D, A, A), tau_f=0.8, tau_T=1.15, Q=1e-4, ax=1e-6), "E"),
    (9, 8, dict(bc=(P, P, D, A), T_bc=(0.0, 0.0, 1.0, 0.0),
                u_bc=((0.0, 0.0), (0.0, 0.0), (0.0, 1e-3), (0.01, 1e-3))), "S"),
    (8, 7, dict(bc=(D, A, P, P), tau_f=1.1, tau_T=0.9), "W"),
    (40, 9, dict(bc=(D, D, D, A), T_bc=(1.0, 0.0, 0.4, 0.0), u_bc=((0.0, 0.0), (0.0, 0.0), (0.0, 0.0), (0.02, 0.0)),
                 tau_f=0.9, Q=1e-5), "W"),
]


@pytest.mark.parametrize("nx,ny,more,side", CASES)
def test_adjoint_matches_oracle_complex_step(nx, ny, more, side):
    steps = 25
    p = W.cavity(nx, 1e4, 1e-2, 0.6, ny=ny, **more)
    eps = W.gaussian_random_field(48, corr=4.0, seed=4)[:ny, :nx]
    g = lbm.Lattice(p, "f64")
    g.set_fields(eps_field=eps)
    loss, g_eps, g_t = g.adjoint(steps, side=side, segment=4)
    cells = sorted({(x, y) for x in (0, 1, 2, nx // 2, nx - 3, nx - 2, nx - 1) for y in (0, 1, 2, ny // 2, ny - 3, ny - 2, ny - 1)})
    walls = [s for s, kind in zip("WESN", p["bc"]) if kind == D]
    ref, ref_t = oracle.nusselt_gradient(p, steps, eps, cells, sides=walls, loss_side=side)
    assert loss == pytest.approx(oracle.Oracle(p, eps_field=eps).run(steps).nusselt(side)[0], rel=1e-12)
    scale = np.abs(ref).max()
    assert scale > 0
    for k, (x, y) in enumerate(cells):
        assert g_eps[y, x] == pytest.approx(ref[k], abs=1e-9 * scale), (x, y)
    for s in walls:
        assert g_t["WESN".index(s)] == pytest.approx(ref_t[s], rel=1e-9, abs=1e-12), s
