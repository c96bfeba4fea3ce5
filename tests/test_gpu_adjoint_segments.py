"""The gradient does not depend on which states are kept: all of them (segment
0 on small runs: in FP32 every second one comes from the middle of a two-step
launch), or checkpoints every `segment` steps with the rest recomputed.  The
same states and the same backward steps: the same bits, at the edges of the
two-step kernel's tiles (62 columns, 6 and 8 rows), for even and odd step
counts, all kinds of sides, relaxation times on and off 1.  And segment 0 against the
oracle's complex-step derivatives."""
import numpy as np
import pytest

import oracle
from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

from test_gpu_two_steps import SIDES

pytestmark = pytest.mark.gpu

LOSS = {"cavity": "W", "mixed": "N", "channel": "S", "shaft": "E"}


def _run(p, fields, eps, precision, steps, segment, side):
    g = lbm.Lattice(p, precision)
    g.set_fields(*fields, eps_field=eps)
    loss, g_eps, g_t = g.adjoint(steps, side=side, segment=segment)
    g.sync()
    g.check_guards()
    m = g.moments()  # the state the run ends in
    return [np.float64(loss), g_eps, g_t, m["T"], m["ux"]]


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("sides", sorted(LOSS))
@pytest.mark.parametrize("nx,ny,tau", [(8, 8, 1.0), (63, 19, 1.0), (131, 40, 0.85), (620, 203, 1.0)])
def test_kept_and_recomputed_states(nx, ny, tau, sides, precision):
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, tau_f=tau, tau_T=tau, Q=1e-5, **SIDES[sides])
    fields = W.random_fields(p, seed=nx, amp_u=1e-3, amp_T=0.1)
    eps = np.random.Generator(np.random.PCG64(nx)).uniform(0.35, 0.85, (ny, nx))
    for steps in (1, 8, 15) if nx < 600 else (5,):
        kept = _run(p, fields, eps, precision, steps, 0, LOSS[sides])
        assert np.abs(kept[1]).max() > 0 and all(np.all(np.isfinite(v)) for v in kept)
        for segment in (1, 7):
            for a, b in zip(kept, _run(p, fields, eps, precision, steps, segment, LOSS[sides])):
                assert np.array_equal(a, b), (steps, segment)


@pytest.mark.parametrize("sides", sorted(LOSS))
def test_kept_states_against_the_oracle(sides):
    n, ny, steps = 13, 12, 41
    p = W.cavity(n, 1e4, 1e-2, 0.6, ny=ny, **SIDES[sides])
    eps = W.gaussian_random_field(16, corr=4.0, seed=4)[:ny, :n]
    g = lbm.Lattice(p, "f64")
    g.set_fields(eps_field=eps)
    loss, g_eps, g_t = g.adjoint(steps, side=LOSS[sides])
    cells = [(0, 0), (1, 1), (6, 0), (12, 11), (6, 5), (11, 2)]
    walls = [s for s, kind in zip("WESN", p["bc"]) if kind == "dirichlet"]
    ref, ref_t = oracle.nusselt_gradient(p, steps, eps, cells, sides=walls, loss_side=LOSS[sides])
    assert loss == pytest.approx(oracle.Oracle(p, eps_field=eps).run(steps).nusselt(LOSS[sides])[0], rel=1e-12)
    scale = np.abs(ref).max()
    assert scale > 0
    for k, (x, y) in enumerate(cells):
        assert g_eps[y, x] == pytest.approx(ref[k], abs=1e-9 * scale), (x, y)
    for s in walls:
        assert g_t["WESN".index(s)] == pytest.approx(ref_t[s], rel=1e-9, abs=1e-12), s
