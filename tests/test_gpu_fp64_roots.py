"""The FP64 square root and reciprocal of the node update (lbm_core.cuh)
against numpy's, over what reaches them: zero, subnormal and the smallest normal
squares of speeds, and sixty powers of two on both sides of 1."""
import ctypes as C
import subprocess

import numpy as np
import pytest
import torch

from paper_1505_02976_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = """
#include "lbm_core.cuh"
__global__ void k_roots(const double* x, double* root, double* inverse, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    root[i] = lbm::lsqrt(x[i]);
    inverse[i] = lbm::lrcp(x[i]);
}
extern "C" int roots(const double* x, double* root, double* inverse, int n) {
    k_roots<<<(n + 255) / 256, 256>>>(x, root, inverse, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    src, lib = d / "roots.cu", d / "roots.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), "-shared", *build.NVCC_FLAGS, "-I", build.CSRC, "-o", str(lib), str(src)], check=True)
    fn = C.CDLL(str(lib)).roots

    def call(x):
        t = torch.from_numpy(np.ascontiguousarray(x, np.float64)).cuda()
        a, b = torch.empty_like(t), torch.empty_like(t)
        torch.cuda.synchronize()
        assert fn(*(C.c_void_p(v.data_ptr()) for v in (t, a, b)), C.c_int(t.numel())) == 0
        return a.cpu().numpy(), b.cpu().numpy()

    return call


def _samples(lo, hi, n, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))


def test_root_of_zero_and_subnormal_values(roots):
    tiny = np.finfo(np.float64).tiny
    x = np.r_[0.0, 5e-324, tiny * np.exp2(-np.arange(1.0, 53.0)), np.nextafter(tiny, 0.0)]
    root, _ = roots(x)
    # below the smallest normal number the root may be 0: |v| < 1.5e-154
    assert np.all((root >= 0.0) & (root <= np.sqrt(x) * (1 + 2.0 ** -52)))


def test_root_and_reciprocal_of_normal_values(roots):
    tiny = np.finfo(np.float64).tiny
    x = np.r_[tiny, np.nextafter(tiny, 1.0), _samples(-1022, 1000, 1 << 20, 1), _samples(-60, 61, 1 << 20, 2)]
    root, inverse = roots(x)
    assert np.all(np.abs(root - np.sqrt(x)) <= np.spacing(np.sqrt(x)))
    assert np.all(np.abs(inverse - 1.0 / x) <= np.spacing(1.0 / x))


def test_root_and_reciprocal_are_rounded_once(roots):
    """At most half a unit in the last place off (and 1e-3 of one), as the language's own."""
    x = np.r_[_samples(-900, 900, 1 << 18, 3), _samples(-4, 5, 1 << 19, 4), np.nextafter(1.0, [0.0, 2.0]), 0.25, 1.0, 2.0, 4.0]
    root, inverse = roots(x)
    wide = x.astype(np.longdouble)
    for got, want in ((root, np.sqrt(wide)), (inverse, 1 / wide)):
        ulp = np.spacing(np.abs(want).astype(np.float64))
        assert np.max(np.abs(got.astype(np.longdouble) - want) / ulp) <= 0.501
