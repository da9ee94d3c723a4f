"""Which kernels a context's Gauss-Newton transport solves run in, by the launches that the kernel
timer counts (class 4: one launch per resident solve; class 0: column kernels of the pairs): the
resident solves by default on grids of 64 to 256 points per axis up to 2^15 points (H2: 2^14), the
kernel pairs on larger ones and where they were asked for, the default again after a reset.  Equal results on all."""
import numpy as np
import pytest

from paper_1503_00757_gb300 import synth

from .gpu_util import to_gpu

pytestmark = pytest.mark.gpu

NT = 2


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("regnorm", [1, 2])
@pytest.mark.parametrize("n1,n2", [(64, 64), (64, 128), (64, 256), (128, 64), (128, 128), (128, 256), (256, 64),
                                   (256, 128), (256, 256), (32, 64)])
def test_default_path_and_the_way_back_to_it(n1, n2, regnorm):
    import torch
    from paper_1503_00757_gb300.binding import Context
    rng = np.random.default_rng(n1 + 3 * n2)
    mT, mR = (to_gpu(synth.rescale01(synth.smooth_field(n1, n2, 4, rng))) for _ in range(2))
    v, vt = (to_gpu(synth.velocity(n1, n2, 4, 0.1, rng, 0.3)) for _ in range(2))
    ctx = Context(n1, n2, NT, regnorm=regnorm, beta=1e-2)
    torch.cuda.synchronize()
    ctx.set_images(mT, mR)
    g, H = torch.empty(2, n1, n2, device="cuda"), torch.empty(2, n1, n2, device="cuda")

    def solves():
        ctx.kernel_timing(True)
        ctx.gradient(v, g)
        ctx.hessian_matvec(vt, H)
        resident, column = ctx.kernel_time(4)[0], ctx.kernel_time(0)[0]
        ctx.kernel_timing(False)
        return resident, column, g.clone(), H.clone()

    small = n1 * n2 <= (2 ** 15 if regnorm == 1 else 2 ** 14) and min(n1, n2) >= 64
    first = solves()
    ctx.set_transport(False)
    pairs = solves()
    ctx.set_transport(None)
    again = solves()
    ctx.close()
    # one launch each for the state, the adjoint and the matvec's two solves, or a column pass per Heun stage
    assert first[0] == again[0] == (3 if small else 0) and pairs[0] == 0
    assert pairs[1] >= 8 * NT - 1 and first[1] == again[1] and (first[1] < pairs[1]) == small
    for o in (pairs, again):
        assert torch.equal(o[2], first[2]) and torch.equal(o[3], first[3])
