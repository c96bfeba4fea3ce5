"""The moment state's kernel over tiles (the default of FP32 lattices up to 16
tiles an SM) against the kernel over bands: the same operations on every node,
so the same bits, at the smallest lattices, tile edges (62 columns, 6 and 8
rows), odd sizes, every kind of side, with a porosity field and a profile."""
import numpy as np
import pytest

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

from test_gpu_two_steps import SIDES

pytestmark = pytest.mark.gpu


def _run(p, fields, steps, segments, eps, ay):
    g = lbm.Lattice(p, "f32", state="moments")
    g.set_moment_segments(segments)
    g.set_fields(*fields, eps_field=eps)
    g.set_force_profile(ay)
    g.step(steps)
    g.sync()
    g.check_guards()
    f, h = g.get_state()
    return f[1:], h


@pytest.mark.parametrize("sides", sorted(SIDES))
@pytest.mark.parametrize("nx,ny,field", [(8, 8, False), (9, 11, True), (62, 18, False), (63, 19, False), (131, 40, True),
                                         (700, 517, False), (1301, 203, True)])
def test_tiles_match_bands(nx, ny, field, sides):
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, Q=1e-5, ax=1e-6, **SIDES[sides])
    fields = W.random_fields(p, seed=nx + ny, amp_u=2e-3, amp_T=0.3)
    eps = None
    if field:
        rng = np.random.Generator(np.random.PCG64(7))
        eps = rng.uniform(0.3, 0.9, (ny, nx))
    ay = 1e-6 * np.arange(ny)
    for steps in (1, 6):
        a, b = _run(p, fields, steps, 0, eps, ay), _run(p, fields, steps, 3, eps, ay)
        assert np.all(np.isfinite(b[1]))
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
