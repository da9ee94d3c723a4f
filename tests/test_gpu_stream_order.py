"""Order between a context's set-up, which uses the legacy default stream, and its first kernels on
a working stream that is not ordered after it (cudaStreamNonBlocking, as torch's streams are)."""
import math

import numpy as np
import pytest

from .gpu_util import to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_3d_context_is_ready_when_created():
    """Its tables are on the device when the constructor returns, so the first gradient, issued at
    once on a non-blocking stream, equals every later one bit for bit."""
    import torch
    from paper_1503_00757_gb300.binding import Context3D
    shape, nt = (16, 32, 64), 1
    rng = np.random.default_rng(11)
    mT, mR = (to_gpu(rng.random(shape)) for _ in range(2))
    v = to_gpu(0.05 * rng.standard_normal((3, *shape)))
    s = torch.cuda.Stream()
    outs = []
    for _ in range(16):
        g, again = torch.empty(3, *shape, device="cuda"), torch.empty(3, *shape, device="cuda")
        torch.cuda.synchronize()
        ctx = Context3D(*shape, nt, beta=1e-2, gamma=math.inf, stream=s)
        idle = torch.cuda.default_stream().query()
        ctx.set_images(mT, mR)
        ctx.gradient(v, g)
        torch.cuda.synchronize()
        outs.append(g)
        ctx.gradient(v, again)
        torch.cuda.synchronize()
        ctx.close()
        assert idle, "the set-up's copy was still in flight"
        assert torch.equal(g, again)
    assert all(torch.equal(outs[0], o) for o in outs[1:])


def test_2d_context_is_ready_when_created():
    """The same for 2-D contexts: the shear model with a mass source reads a scalar that the
    constructor uploads last."""
    import torch
    from paper_1503_00757_gb300.binding import Context
    n, nt = 32, 1
    rng = np.random.default_rng(12)
    mT, mR = (to_gpu(rng.random((n, n))) for _ in range(2))
    v = to_gpu(0.05 * rng.standard_normal((2, n, n)))
    s = torch.cuda.Stream()
    outs = []
    for _ in range(16):
        g, again = torch.empty(2, n, n, device="cuda"), torch.empty(2, n, n, device="cuda")
        torch.cuda.synchronize()
        ctx = Context(n, n, nt, beta=1e-2, gamma=1e-3, shear=0.5, stream=s)
        idle = torch.cuda.default_stream().query()
        ctx.set_images(mT, mR)
        ctx.gradient(v, g)
        ctx.gradient(v, again)
        torch.cuda.synchronize()
        ctx.close()
        assert idle, "the set-up's copy was still in flight"
        assert torch.equal(g, again)
        outs.append(g)
    assert all(torch.equal(outs[0], o) for o in outs[1:])
