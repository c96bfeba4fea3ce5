"""The FP64 one-step kernel where its blocks come in two and three rounds of one
size, at their edges (12 to 37 blocks of one warp on each of 152 SMs), bit for
bit against the batched kernel in another launch shape, at relaxation times on
and off 1."""
import numpy as np
import pytest

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [dict(), dict(tau_f=0.8, tau_T=1.15)])
@pytest.mark.parametrize("ny", [880, 885, 900, 1100, 1320, 1330, 1400, 1768, 1775, 1900, 2200, 2215, 2650])
def test_fp64_step_in_rounds(ny, tau):
    p = W.cavity(40, 1e5, 1e-3, 0.5, ny=ny, **tau)
    fields = W.random_fields(p, seed=ny, amp_u=1e-3)
    g = lbm.Lattice(p, "f64")
    g.set_fields(*fields)
    g.step(3)
    b = lbm.Batch([p], "f64")
    b.set_fields(0, *fields)
    b.step(3)
    m, mb = g.moments(), b.moments(0)
    for k in ("p", "ux", "uy", "T"):
        assert np.array_equal(m[k], mb[k]), k
