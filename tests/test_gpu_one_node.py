"""The stream function of the smallest lattices: one node (whose scratch is
larger than its fields), one column, one row."""
import numpy as np
import pytest

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 1), (1, 2), (1, 65), (300, 1)])
def test_stream_function(nx, ny, precision):
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, bc=("periodic",) * 4, L=8.0)
    g = lbm.Lattice(p, precision)
    T, ux, uy = W.random_fields(p, seed=1, amp_u=1e-2)
    g.set_fields(T, ux, uy)
    psi, (lo, hi) = g.stream_function()
    g.check_guards()
    u = g.moments()["ux"]
    want = np.concatenate([np.zeros((1, nx)), np.cumsum(0.5 * (u[1:] + u[:-1]), axis=0)])
    assert np.abs(psi - want).max() <= 1e-14 * ny
    assert lo == psi.min() and hi == psi.max()
