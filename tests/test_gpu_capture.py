"""Calls made while a caller captures a CUDA graph: on the stream that is being captured, and on
other streams meanwhile."""
import math

import numpy as np
import pytest

from paper_1503_00757_gb300 import synth

from .gpu_util import to_gpu

pytestmark = pytest.mark.gpu

N, NT = 64, 3


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _inputs():
    rng = np.random.default_rng(5)
    mT, mR = (synth.rescale01(synth.smooth_field(N, N, 4, rng)) for _ in range(2))
    return [to_gpu(x) for x in (mT, mR, synth.velocity(N, N, 4, 0.2, rng, 0.3), synth.velocity(N, N, 4, 0.2, rng, 0.3))]


@pytest.mark.parametrize("regnorm", [1, 2])
@pytest.mark.parametrize("called_before", [False, True])
def test_displacement_inside_a_callers_capture(regnorm, called_before):
    import torch
    from paper_1503_00757_gb300.binding import Context
    _, _, v, w = _inputs()
    s = torch.cuda.Stream()
    ctx = Context(N, N, NT, regnorm=regnorm, stream=s)
    x, u = v.clone(), torch.empty(2, N, N, device="cuda")
    torch.cuda.synchronize()
    if called_before:
        ctx.displacement(x, u)
        torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        ctx.displacement(x, u)
    x.copy_(w)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    replayed = u.clone()
    ctx.displacement(x, u)
    torch.cuda.synchronize()
    ctx.close()
    assert torch.equal(u, replayed)
