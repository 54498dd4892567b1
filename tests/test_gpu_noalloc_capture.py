"""hom_apply_noalloc captured in a CUDA graph: its programmatic launches replay to the bits of a
direct call, at lengths of the register engine and of the runtime one, and to the oracle's operator."""
import numpy as np
import pytest

import oracle
import rve_inputs as ri
from gpu_util import FP32_TOL, rel_maxerr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deriv", [0, 1])
@pytest.mark.parametrize("shape", [(32, 32, 32), (64, 4, 2), (5, 9, 18), (30, 8, 64), (2, 2, 2)])
def test_noalloc_replays(shape, deriv):
    import torch
    from paper_2110_00733_gb300 import build, hom
    build.build()
    hom.load_library()
    phi = torch.tensor(ri.random_phi(shape, 3), dtype=torch.float32, device="cuda")
    eps = torch.tensor(ri.random_field(shape, 4), dtype=torch.float32, device="cuda")
    out = torch.zeros_like(eps)
    s = torch.cuda.Stream()

    def call(o):
        hom.hom_apply_noalloc(shape, phi, eps, o, 1.0, 0.3, deriv, stream=s.cuda_stream)

    torch.cuda.synchronize()
    call(out)
    s.synchronize()
    ref = oracle.apply(phi.double().cpu().numpy(), 1.0, 0.3, deriv, eps.double().cpu().numpy())
    assert rel_maxerr(out.cpu().numpy(), ref) <= FP32_TOL
    again = torch.zeros_like(eps)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        call(again)
        call(again)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, again)
