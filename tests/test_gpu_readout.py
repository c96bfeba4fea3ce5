"""Read-out kernels at the sizes where they can go wrong: the chunked stream
function (32 rows a chunk, 128 columns a block) against numpy's running
trapezoid sum of the GPU's own u_x, FP64 (both sum the same terms in another
order: 1e-14 of the largest |psi|, as for the one-column form); device outputs
written in place or, where they overlap, copied in order; the residual's four
sums against numpy (FP64, 1e-12)."""
import numpy as np
import pytest
import torch

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(5, 4), (128, 31), (129, 32), (7, 33), (130, 64), (40, 257)])
def test_stream_function_chunks(nx, ny):
    p = W.cavity(nx, 1e4, 1e-2, 0.6, ny=ny)
    g = lbm.Lattice(p, "f64")
    g.set_fields(*W.random_fields(p, seed=nx, amp_u=1e-3))
    g.step(3)
    u = g.moments()["ux"]
    psi, (lo, hi) = g.stream_function()
    want = np.concatenate([np.zeros((1, nx)), np.cumsum(0.5 * (u[1:] + u[:-1]), axis=0)])
    assert np.abs(psi - want).max() <= 1e-14 * np.abs(want).max()
    assert lo == psi.min() and hi == psi.max()
    g.check_guards()


@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
def test_device_outputs_in_place_and_overlapping(precision):
    p = W.cavity(40, 1e4, 1e-2, 0.6, ny=30)
    n = 40 * 30
    g = lbm.Lattice(p, precision)
    g.set_fields(*W.random_fields(p, seed=3, amp_u=1e-3))
    g.step(4)
    m = g.moments()
    some = {"T": torch.zeros(n, dtype=torch.float64, device="cuda")}
    g.moments_device(some)
    g.sync()
    assert np.array_equal(some["T"].cpu().numpy().reshape(30, 40), m["T"])
    # ux starts halfway through p: it is copied after p, as uy and T are after it
    buf = torch.zeros(4 * n, dtype=torch.float64, device="cuda")
    g.moments_device({"p": buf[:n], "ux": buf[n // 2:n // 2 + n], "uy": buf[2 * n:3 * n], "T": buf[3 * n:]})
    g.sync()
    got = buf.cpu().numpy()
    assert np.array_equal(got[:n // 2], m["p"].ravel()[:n // 2])
    assert np.array_equal(got[n // 2:n // 2 + n], m["ux"].ravel())
    assert np.array_equal(got[2 * n:3 * n], m["uy"].ravel()) and np.array_equal(got[3 * n:], m["T"].ravel())


@pytest.mark.parametrize("nx,ny", [(4, 4), (31, 9), (200, 131), (700, 517)])
def test_residual_sums(nx, ny):
    p = W.cavity(nx, 1e4, 1e-2, 0.6, ny=ny)
    g = lbm.Lattice(p, "f64")
    g.set_fields(*W.random_fields(p, seed=ny, amp_u=1e-3))
    old = g.moments()  # the snapshot of lbm_set_fields
    g.step(5)
    new = g.moments()
    ru, rT = g.residual()
    du = np.hypot(new["ux"] - old["ux"], new["uy"] - old["uy"]).sum() / np.hypot(new["ux"], new["uy"]).sum()
    dT = np.abs(new["T"] - old["T"]).sum() / np.abs(new["T"]).sum()
    assert ru == pytest.approx(du, rel=1e-12) and rT == pytest.approx(dT, rel=1e-12)
