"""A context's launch sequences run directly at first, then are captured and replayed (csrc/api.cu,
run_seq): every call gives the same result on the default stream and on a working stream, also after
parameters changed (which drops the captures) and with buffers that change from call to call."""
import math

import numpy as np
import pytest

from paper_1503_00757_gb300 import synth

from .gpu_util import to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("working_stream", [False, True])
@pytest.mark.parametrize("n,regnorm,shear", [(32, 1, 0.0), (32, 2, 0.0), (64, 1, 0.0), (64, 2, 0.0), (32, 1, 0.5)])
def test_every_call_of_a_sequence_gives_the_same_result(n, regnorm, shear, working_stream):
    import torch
    from paper_1503_00757_gb300.binding import Context
    nt, beta = 2, 1e-2
    rng = np.random.default_rng(n + regnorm)
    mT, mR = (to_gpu(synth.rescale01(synth.smooth_field(n, n, 4, rng))) for _ in range(2))
    v, vt = (to_gpu(synth.velocity(n, n, 4, 0.2, rng, 0.3)) for _ in range(2))
    lT, lR = (mT > 0.5).float(), (mR > 0.5).float()
    ctx = Context(n, n, nt, regnorm=regnorm, beta=beta, gamma=1e-3, shear=shear,
                  stream=torch.cuda.Stream() if working_stream else None)
    torch.cuda.synchronize()
    ctx.set_images(mT, mR)

    def once():
        # buffers of this call's own (kept: no two calls share an address)
        E = lambda k: torch.full((k, n, n), float("nan"), device="cuda")
        m1, g, H, u, det, lab = E(1), E(2), E(2), E(2), E(1), E(1)
        a, b = v.clone(), vt.clone()
        torch.cuda.synchronize()
        J1, J2 = ctx.objective(a, m1), ctx.gradient(a, g)
        ctx.hessian_matvec(b, H)
        ctx.hessian_matvec(b, b)  # in place
        ctx.displacement(a, u)
        ctx.label_overlap(a, lT, lR, lab)
        s = ctx.detgrad(a, det)
        torch.cuda.synchronize()
        assert torch.equal(b, H)
        return (m1, g, H, u, lab, det), (J1, J2, s), (a, b)

    calls = [once() for _ in range(13)]
    ctx.set_params(nt + 1, regnorm, 2 * beta, math.inf, shear)
    other = once()
    ctx.set_params(nt, regnorm, beta, 1e-3, shear)
    calls += [once() for _ in range(2)]
    ctx.close()
    for c in calls[1:]:
        assert all(torch.equal(x, y) for x, y in zip(c[0], calls[0][0]))
        assert c[1] == calls[0][1]
    assert not torch.equal(other[0][1], calls[0][0][1])
    assert all(bool(torch.isfinite(x).all()) for x in calls[0][0] + other[0])
