"""A user's own CUDA graph around the asynchronous calls: new fields from
device tensors, steps, and the moment fields to device tensors, captured once
and replayed on new values in the same tensors, against the same calls made
directly (the same bits)."""
import numpy as np
import pytest
import torch

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W

from test_gpu_two_steps import SIDES

pytestmark = pytest.mark.gpu

NAMES = ("p", "ux", "uy", "T")


@pytest.mark.parametrize("sides", ["cavity", "channel"])
@pytest.mark.parametrize("precision,state", [("f32", "populations"), ("f64", "populations"), ("f16", "populations"),
                                             ("f32", "moments"), ("f64", "moments")])
def test_fields_steps_and_moments_in_a_graph(precision, state, sides):
    nx, ny = 150, 97
    p = W.cavity(nx, 1e5, 1e-3, 0.5, ny=ny, **SIDES[sides])
    eps = torch.from_numpy(np.random.Generator(np.random.PCG64(1)).uniform(0.3, 0.9, (ny, nx))).cuda()
    inputs = [[torch.from_numpy(v).cuda() for v in W.random_fields(p, seed=s, amp_u=1e-3)] for s in (1, 2)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        g = lbm.Lattice(p, precision, state=state, stream=stream)
        out = {k: torch.empty(ny, nx, dtype=torch.float64, device="cuda") for k in NAMES}
        fields = [torch.empty_like(v) for v in inputs[0]]

        def calls():
            g.set_fields(*fields, eps_field=eps)
            g.step(5)
            g.moments_device(out)

        want = []
        for given in inputs:
            for f, v in zip(fields, given):
                f.copy_(v)
            calls()
            want.append({k: out[k].clone() for k in NAMES})
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            calls()
        for given, ref in zip(inputs, want):
            for f, v in zip(fields, given):
                f.copy_(v)
            for k in NAMES:
                out[k].zero_()
            graph.replay()
            stream.synchronize()
            for k in NAMES:
                assert torch.equal(out[k], ref[k]), k
    assert not torch.equal(want[0]["T"], want[1]["T"])
