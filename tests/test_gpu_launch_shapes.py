"""The FP64 one-step kernel at every share of blocks per SM its launch rule
distinguishes (2 column blocks and a perimeter: 1 to 14 blocks of one warp on
each of 152 SMs), bit for bit against the batched kernel, which runs the same
per-node code in another launch shape."""
import numpy as np
import pytest

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [40, 140, 210, 257, 290, 330, 370, 440, 520, 600, 680, 760, 840, 900, 1000])
def test_fp64_step_at_every_share_of_blocks(ny):
    p = W.cavity(40, 1e5, 1e-3, 0.5, ny=ny)
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
