"""The step-kernel switch off and on again: an FP32 lattice that cannot stage
rows (a periodic side) returns to two steps per launch, and 1 stays refused
where there is nothing to return to."""
import numpy as np
import pytest

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _launches(g, steps):
    before = g.launches
    g.step(steps)
    g.sync()
    return g.launches - before


@pytest.mark.parametrize("p", [W.poiseuille(nx=16, ny=32), W.cavity(20, 1e5, 1e-3, 0.5, bc=("periodic",) * 4),
                               W.cavity(33, 1e5, 1e-3, 0.5)])
def test_off_and_on_again(p):
    walled = "periodic" not in p["bc"]
    g, ref = lbm.Lattice(p, "f32"), lbm.Lattice(p, "f32")
    assert _launches(g, 6) == 3
    g.staged = False
    assert _launches(g, 6) == 6 and not g.staged
    g.staged = True
    assert g.staged == walled and _launches(g, 6) == 3
    if not walled:
        with pytest.raises(lbm.LbmError):
            g.staged = True
        assert _launches(g, 2) == 1
    ref.step(g.steps)
    assert np.array_equal(g.moments()["T"], ref.moments()["T"])


@pytest.mark.parametrize("p,precision,state", [
    (W.poiseuille(nx=6, ny=32), "f32", "populations"),  # too narrow for pairs
    (W.cavity(32, 1e5, 1e-3, 0.5), "f64", "populations"),
    (W.cavity(32, 1e5, 1e-3, 0.5), "f32", "moments"),
    (W.cavity(32, 1e5, 1e-3, 0.5, bc=("periodic",) * 4), "f16", "populations")])
def test_on_stays_refused_after_off(p, precision, state):
    g = lbm.Lattice(p, precision, state=state)
    g.staged = False
    with pytest.raises(lbm.LbmError):
        g.staged = True
    assert not g.staged and _launches(g, 2) == 2
