"""FP32 lattices at relaxation times off 1 give the same bits however their
steps are cut into calls: pairs of steps, single steps and the kernels that take
them (two steps from shared memory, staged rows, global loads) run the same
operations, at the walls too.  Sizes at the edges of a tile (62 columns, 6 or
8 rows) and of both launch shapes; a run resumed from a checkpoint after an odd
number of steps; batches in every mode; and FP16 storage with either kernel."""
import numpy as np
import pytest

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

from test_gpu_two_steps import SIDES

pytestmark = pytest.mark.gpu

TAU = dict(tau_f=0.8, tau_T=1.15, Q=1e-5, ax=1e-6)


def _problem(nx, ny, sides, field):
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, **TAU, **SIDES[sides])
    eps = None
    if field:
        eps = np.random.Generator(np.random.PCG64(nx)).uniform(0.3, 0.9, (ny, nx))
    return p, W.random_fields(p, seed=nx + ny, amp_u=2e-3, amp_T=0.3), eps


def _run(p, fields, eps, calls, staged=True, ay=None):
    g = lbm.Lattice(p, "f32")
    g.set_fields(*fields, eps_field=eps)
    if ay is not None:
        g.set_force_profile(ay)
    if not staged:
        g.staged = False
    for n in calls:
        g.step(n)
    g.sync()
    f, h = g.get_state()
    return np.concatenate([f[1:], h])


@pytest.mark.parametrize("sides", sorted(SIDES))
@pytest.mark.parametrize("nx,ny,field", [(8, 8, False), (9, 11, True), (62, 18, False), (63, 19, True), (131, 40, False),
                                         (1301, 203, True)])
def test_calls_cut_anywhere(nx, ny, sides, field):
    p, fields, eps = _problem(nx, ny, sides, field)
    ay = 1e-6 * np.arange(ny)
    whole = _run(p, fields, eps, [7], ay=ay)
    assert np.all(np.isfinite(whole))
    for calls, staged in (([1] * 7, True), ([1, 4, 2], True), ([7], False)):
        assert np.array_equal(whole, _run(p, fields, eps, calls, staged, ay)), (calls, staged)


@pytest.mark.parametrize("sides", ["cavity", "shaft"])
def test_a_resumed_run(tmp_path, sides):
    p, fields, eps = _problem(130, 41, sides, False)
    g = lbm.Lattice(p, "f32")
    g.set_fields(*fields)
    g.step(5)
    g.save(str(tmp_path / "state"))
    r = lbm.Lattice(p, "f32")
    r.load_checkpoint(str(tmp_path / "state"))
    r.step(6)
    r.sync()
    f, h = r.get_state()
    assert np.array_equal(np.concatenate([f[1:], h]), _run(p, fields, eps, [11]))


def test_batches():
    probs = [_problem(nx, ny, s, False) for nx, ny, s in ((20, 31, "cavity"), (130, 50, "mixed"), (64, 64, "cavity"))]
    runs = []
    for mode, calls, staged in (("fused", [9], True), ("fused", [1] * 9, True), ("per_case", [9], True),
                                ("persistent", [4, 5], True), ("fused", [9], False)):
        b = lbm.Batch([p for p, _, _ in probs], "f32")
        b.staged = staged
        for c, (_, fields, _) in enumerate(probs):
            b.set_fields(c, *fields)
        for n in calls:
            b.step(n, mode)
        b.sync()
        runs.append([b.moments(c) for c in range(len(probs))])
    for other in runs[1:]:
        for a, m in zip(runs[0], other):
            assert all(np.array_equal(a[k], m[k]) for k in ("p", "ux", "uy", "T"))


@pytest.mark.parametrize("tau", [dict(), TAU])
@pytest.mark.parametrize("nx,ny,field", [(300, 50, False), (129, 131, True), (517, 9, False), (4, 4, False)])
def test_fp16_kernels(nx, ny, field, tau):
    """FP16 storage: node pairs from staged rows and single nodes from global memory."""
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, **tau, **SIDES["mixed"])
    eps = np.random.Generator(np.random.PCG64(nx)).uniform(0.3, 0.9, (ny, nx)) if field else None
    fields = W.random_fields(p, seed=nx + ny, amp_u=2e-3, amp_T=0.3)
    states = []
    for staged in (True, False):
        g = lbm.Lattice(p, "f16")
        g.set_fields(*fields, eps_field=eps)
        g.staged = staged
        g.step(30)
        g.sync()
        f, h = g.get_state()
        states.append(np.concatenate([f[1:], h]))
    assert np.array_equal(states[0], states[1])
