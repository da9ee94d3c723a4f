"""Three-dimensional transport through axis-wise derivatives (csrc/deriv.cuh, csrc/reg3d.cu) at the
sizes where its launch rules change: the smallest box, one column block per axis; the box sizes at
which the column and row blocks grow (2^17, 2^18, 2^20 points) and axes of 128 and 256 points take 16 entries a thread; columns
shorter than a block.

Tolerance as in test_gpu_reg3d: max(1, c) (2e-5 + 2 u (n / 2) log2(n)), n the longest axis, c the
conditioning of the sums g and H v~."""
import math

import numpy as np
import pytest

from oracle import reg3d as R

from .gpu_util import check, to_gpu, to_np
from .test_gpu_reg3d import _inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("shape,nt,beta_w", [
    ((8, 8, 8), 1, math.inf), ((8, 16, 8), 2, 0.0), ((64, 64, 32), 1, 1e-3), ((32, 64, 128), 1, math.inf),
    ((64, 128, 128), 1, 1e-3), ((256, 128, 32), 1, math.inf),
])
def test_block_size_edges_match_oracle(shape, nt, beta_w):
    import torch
    from paper_1503_00757_gb300.binding import Context3D
    beta = 1e-2
    mT, mR, v, vt = _inputs(shape, 7300 + sum(shape) + nt, nt)
    P = R.Registration3D(mT, mR, nt, beta, beta_w)
    g_ref, J_ref = P.gradient(v)
    H_ref = P.matvec(vt)
    outs = []
    for stream in (None, torch.cuda.Stream()):
        ctx = Context3D(*shape, nt, beta=beta, gamma=beta_w, stream=stream)
        ctx.set_images(to_gpu(mT), to_gpu(mR))
        vg, vtg = to_gpu(v), to_gpu(vt)
        torch.cuda.synchronize()
        g, H = torch.empty(3, *shape, device="cuda"), torch.empty(3, *shape, device="cuda")
        J = ctx.gradient(vg, g)
        ctx.hessian_matvec(vtg, H)
        torch.cuda.synchronize()
        ctx.close()
        outs.append((g, H, J))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1]) and outs[0][2] == outs[1][2]
    g, H, J = outs[0]
    tag = f"{shape} nt={nt} beta_w={beta_w}"
    n = max(shape)
    base = 2e-5 + 2.0 * 2.0 ** -24 * (n / 2) * math.log2(n)
    check(f"3-D J ({tag})", abs(J - J_ref) / abs(J_ref), 2e-5)
    c_g = (R.norm(beta * R.apply_A(v)) + R.norm(P.b)) / R.norm(g_ref)
    check(f"3-D gradient ({tag})", np.linalg.norm(to_np(g) - g_ref) / np.linalg.norm(g_ref), base * max(1.0, c_g),
          cond=c_g)
    c_h = (R.norm(beta * R.apply_A(vt)) + R.norm(P.bt)) / R.norm(H_ref)
    check(f"3-D Gauss-Newton matvec ({tag})", np.linalg.norm(to_np(H) - H_ref) / np.linalg.norm(H_ref),
          base * max(1.0, c_h), cond=c_h)


def test_matvec_inside_a_callers_capture():
    """The matvec's launch sequence goes into a graph the caller is capturing, and replays with new inputs."""
    import torch
    from paper_1503_00757_gb300.binding import Context3D
    shape, nt = (16, 16, 32), 3
    mT, mR, v, vt = _inputs(shape, 7400, nt)
    s = torch.cuda.Stream()
    ctx = Context3D(*shape, nt, beta=1e-2, stream=s)
    ctx.set_images(to_gpu(mT), to_gpu(mR))
    x, H, g = to_gpu(vt), torch.empty(3, *shape, device="cuda"), torch.empty(3, *shape, device="cuda")
    torch.cuda.synchronize()
    ctx.gradient(to_gpu(v), g)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        ctx.hessian_matvec(x, H)
    x.copy_(to_gpu(0.5 * vt + 0.1))
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    replayed = H.clone()
    ctx.hessian_matvec(x, H)
    torch.cuda.synchronize()
    ctx.close()
    assert torch.equal(H, replayed)
