"""The full-Newton variants of the axis-wise adjoint kernels (csrc/transport.cu: second product of the
column kernel, k_adj_row with the adjoint history) on unequal axes and on lines of 16 to 1024 points.

At a residual of exactly zero (the reference is the transported template, bit for bit) the adjoint
history is zero, and the full-Newton matvec has to be the Gauss-Newton one: its extra terms add exact
zeros, and the variants do the same arithmetic in the same order.  Values at a nonzero residual are
compared with the oracle in test_gpu_full_newton."""
import numpy as np
import pytest

from paper_1503_00757_gb300 import synth

from .gpu_util import make_ctx, to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("n1,n2,nt", [(16, 16, 1), (16, 32, 2), (256, 64, 4), (64, 512, 3), (1024, 32, 2), (32, 1024, 2),
                                      (256, 256, 4), (1024, 1024, 1)])
def test_full_newton_is_gauss_newton_at_zero_residual(n1, n2, nt):
    import torch
    rng = np.random.default_rng(n1 + 5 * n2)
    mT = to_gpu(synth.rescale01(synth.smooth_field(n1, n2, 2, rng)))
    v, vt = (to_gpu(synth.velocity(n1, n2, 2, 0.2 * 6.28 * nt / max(n1, n2), rng, grad_fraction=0.3)) for _ in range(2))
    E = lambda k: torch.empty(k, n1, n2, device="cuda")
    outs = []
    for full in (False, True):
        ctx = make_ctx(n1, n2, nt, beta=1e-3, gamma=1e-3)
        ctx.set_transport(False)
        ctx.set_hessian(full)
        m1, g, H, b = E(1), E(2), E(2), E(2)
        ctx.set_images(mT, mT)
        ctx.objective(v, m1)
        ctx.set_images(mT, m1[0])
        ctx.gradient(v, g)
        ctx.body_force(b)
        assert not bool(b.any())
        ctx.hessian_matvec(vt, H)
        ctx.body_force(b)
        torch.cuda.synchronize()
        ctx.close()
        assert bool(b.any()) and bool(torch.isfinite(H).all())
        outs.append((g, H, b))
    assert all(torch.equal(x, y) for x, y in zip(*outs))
