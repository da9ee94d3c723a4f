"""Transport by axis-wise derivatives (csrc/transport.cu, csrc/transport_resident.cu) at the sizes
where a kernel or a launch rule changes: the smallest and the most anisotropic grids, 1024-point
rows (one kernel variant), odd and single time steps; the resident solves of 64- to 256-point grids
against the kernel pairs, which do the same arithmetic in the same order (equal bit for bit);
gradient and divergence with overlapping buffers.

Tolerances: spectral derivatives 1e-5 and J 1e-5 relative to FP64 as in test_gpu_parity; m(1)
1e-5; g and H v~ by that file's op_tol (FP32 rounding of the sums)."""
import math

import numpy as np
import pytest

from oracle import spectral as S
from oracle import transport as T
from oracle.registration import Registration
from paper_1503_00757_gb300 import synth

from .gpu_util import check_rel, to_gpu, to_np
from .test_gpu_parity import OP_TOL, op_cond, op_tol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _problem(n1, n2, seed, vmax):
    rng = np.random.default_rng(seed)
    k = min(4, n1 // 4 - 1, n2 // 4 - 1)
    mT = synth.rescale01(synth.smooth_field(n1, n2, k, rng))
    mR = synth.rescale01(synth.smooth_field(n1, n2, k, rng))
    return mT, mR, synth.velocity(n1, n2, k, vmax, rng, grad_fraction=0.3), synth.velocity(n1, n2, k, 0.3, rng, 0.3)


@pytest.mark.parametrize("n1,n2,nt", [(16, 16, 1), (16, 1024, 2), (1024, 16, 2), (32, 64, 3), (64, 64, 1), (64, 256, 3),
                                      (256, 64, 2), (128, 128, 5), (512, 64, 2)])
def test_gradient_and_matvec_at_grid_edges(n1, n2, nt):
    import torch
    from paper_1503_00757_gb300.binding import Context
    mT, mR, v, vt = _problem(n1, n2, n1 + 3 * n2 + nt, min(0.3, 0.25 * 2 * math.pi * nt / max(n1, n2)))
    P = Registration(mT, mR, nt, regnorm=1, beta_v=1e-2, beta_w=1e-3)
    g_ref, J_ref = P.gradient(v)
    b_ref = P.b
    H_ref = P.matvec(vt)
    ctx = Context(n1, n2, nt, regnorm=1, beta=1e-2, gamma=1e-3)
    ctx.set_images(to_gpu(mT), to_gpu(mR))
    g, H = torch.empty(2, n1, n2, device="cuda"), torch.empty(2, n1, n2, device="cuda")
    J = ctx.gradient(to_gpu(v), g)
    ctx.hessian_matvec(to_gpu(vt), H)
    ctx.close()
    tag = f"{n1}x{n2} nt={nt}"
    assert abs(J - J_ref) <= OP_TOL * abs(J_ref)
    check_rel(f"g ({tag})", to_np(g), g_ref, op_tol(1e-2, 1, n1, n2, v, g_ref, b_ref), cond=op_cond(1e-2, 1, v, g_ref, b_ref))
    check_rel(f"H v~ ({tag})", to_np(H), H_ref, op_tol(1e-2, 1, n1, n2, vt, H_ref, P.bt),
              cond=op_cond(1e-2, 1, vt, H_ref, P.bt))


@pytest.mark.parametrize("n1,n2,nt,gamma,shear", [
    (64, 64, 3, 1e-3, "H2"), (64, 128, 1, math.inf, "H2"), (64, 256, 2, 0.0, "H3"), (128, 64, 2, 1e-3, "H2"),
    (128, 128, 5, math.inf, "H2"), (128, 256, 2, 1e-3, "H2"), (256, 64, 3, math.inf, "H3"), (256, 128, 2, 0.0, "H2"),
    (64, 64, 1, 0.0, 0.0), (64, 128, 4, 1e-3, 0.0), (64, 256, 3, math.inf, 0.0), (128, 64, 2, math.inf, 0.5),
    (128, 128, 7, 1e-3, 0.0), (128, 256, 2, 0.0, 0.0), (256, 64, 3, math.inf, 0.0), (256, 128, 2, 1e-3, -0.5),
    (256, 256, 5, math.inf, 0.0)])
def test_resident_solves_equal_the_kernel_pairs(n1, n2, nt, gamma, shear):
    import torch
    from paper_1503_00757_gb300.binding import Context
    mT, mR, v, vt = _problem(n1, n2, 7 * n1 + n2, min(0.3, 0.25 * 2 * math.pi * nt / max(n1, n2)))
    mTd, mRd, vd, vtd = (to_gpu(x) for x in (mT, mR, v, vt))
    torch.cuda.synchronize()
    outs = []
    for resident in (True, False):
        for stream in (None, torch.cuda.Stream()):
            norm = {"H2": 2, "H3": 3}.get(shear, 1)  # the seminorms that keep the spectral stages
            ctx = Context(n1, n2, nt, regnorm=norm, beta=1e-3, gamma=gamma, shear=shear if norm == 1 else 0.0,
                          stream=stream)
            if not resident:
                ctx.set_transport(False)
            ctx.set_images(mTd, mRd)
            g, H, m1, b = (torch.empty(k, n1, n2, device="cuda") for k in (2, 2, 1, 2))
            torch.cuda.synchronize()
            ctx.objective(vd, m1)
            J = ctx.gradient(vd, g)
            ctx.hessian_matvec(vtd, H)
            ctx.body_force(b)
            torch.cuda.synchronize()
            ctx.close()
            outs.append((g, H, m1, b, J))
    for o in outs[1:]:
        assert all(torch.equal(x, y) for x, y in zip(o[:4], outs[0][:4]))
        assert abs(o[4] - outs[0][4]) <= 1e-12 * abs(outs[0][4])


@pytest.mark.parametrize("n1,n2", [(16, 16), (16, 1024), (1024, 16), (64, 32), (512, 1024)])
def test_gradient_and_divergence(n1, n2):
    import torch
    from paper_1503_00757_gb300.binding import Context
    rng = np.random.default_rng(n1 * 3 + n2)
    f, u = rng.standard_normal((n1, n2)), rng.standard_normal((2, n1, n2))
    ctx = Context(n1, n2, 1)
    out, d = torch.empty(2, n1, n2, device="cuda"), torch.empty(n1, n2, device="cuda")
    ctx.spectral_grad(to_gpu(f), out)
    ctx.spectral_div(to_gpu(u), d)
    f32, u32 = f.astype(np.float32).astype(np.float64), u.astype(np.float32).astype(np.float64)
    check_rel(f"grad ({n1}x{n2})", to_np(out), S.grad(f32), OP_TOL)
    check_rel(f"div ({n1}x{n2})", to_np(d), S.div(u32), OP_TOL)
    # the input inside the output buffer
    both = torch.empty(2, n1, n2, device="cuda")
    both[1].copy_(to_gpu(f))
    ctx.spectral_grad(both[1], both)
    uu = to_gpu(u).clone()
    ctx.spectral_div(uu, uu[0])
    torch.cuda.synchronize()
    ctx.close()
    assert torch.equal(both, out) and torch.equal(uu[0], d)


@pytest.mark.parametrize("n1,n2,nt", [(16, 16, 1), (64, 1024, 2), (128, 32, 3)])
def test_deformation_gradient_and_displacement(n1, n2, nt):
    import torch
    from paper_1503_00757_gb300.binding import Context
    _, _, v, _ = _problem(n1, n2, n1 + n2, min(0.3, 0.25 * 2 * math.pi * nt / max(n1, n2)))
    ctx = Context(n1, n2, nt)
    det, u = torch.empty(n1, n2, device="cuda"), torch.empty(2, n1, n2, device="cuda")
    stats = ctx.detgrad(to_gpu(v), det)
    ctx.displacement(to_gpu(v), u)
    torch.cuda.synchronize()
    ctx.close()
    d_ref, D_ref = T.defgrad_measures(T.defgrad_solve(v, nt))
    check_rel("det F1", to_np(det), d_ref, OP_TOL)
    for got, ref in zip(stats, (d_ref.min(), d_ref.mean(), d_ref.max(), D_ref.max(), D_ref.mean())):
        assert abs(got - ref) <= OP_TOL * max(1.0, abs(ref))
    check_rel("displacement", to_np(u), T.displacement_solve(v, nt), OP_TOL)
