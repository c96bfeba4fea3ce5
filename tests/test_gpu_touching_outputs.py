"""Moment fields read out into host arrays that touch: all pageable, each in a
page-locked registration of its own, or some of them."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N, PAGE, NAMES = 128, 4096, ("p", "ux", "uy", "T")
FIELD = N * N * 8
assert FIELD % PAGE == 0


@pytest.mark.parametrize("registered", [(), (0,), (1, 3), (0, 1), (2, 3), (0, 1, 2, 3)])
@pytest.mark.parametrize("kind", ["lattice", "batch"])
def test_fields_that_touch(kind, registered):
    p = W.cavity(N, 1e5, 1e-3, 0.5)
    raw = np.zeros(4 * FIELD + PAGE, np.uint8)
    at = -raw.ctypes.data % PAGE
    out = raw[at:at + 4 * FIELD].view(np.float64).reshape(4, N, N)
    addr = [C.c_void_p(out[q].ctypes.data) for q in range(4)]
    if kind == "lattice":
        g = lbm.Lattice(p, "f32")
        fetch = lambda: g.lib.lbm_moments(g.h, *addr, 0)  # noqa: E731
        ref = lambda: g.moments()  # noqa: E731
    else:
        g = lbm.Batch([p], "f32")
        fetch = lambda: g.lib.lbm_batch_moments(g.h, 0, *addr)  # noqa: E731
        ref = lambda: g.moments(0)  # noqa: E731
    g.step(4)
    g.sync()
    want = ref()
    rt = torch.cuda.cudart()
    for q in registered:
        assert int(rt.cudaHostRegister(addr[q].value, FIELD, 0)) == 0
    try:
        assert fetch() == lbm.LBM_OK
    finally:
        for q in registered:
            assert int(rt.cudaHostUnregister(addr[q].value)) == 0
    for q, k in enumerate(NAMES):
        assert np.array_equal(out[q], want[k]), k
