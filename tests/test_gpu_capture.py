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


@pytest.mark.parametrize("working_stream", [False, True])
def test_first_calls_while_another_stream_is_captured(working_stream):
    """A context's first calls, which capture and instantiate its launch sequences, neither fail nor
    spoil a capture on another stream in the default (global) mode; the results are the usual ones."""
    import ctypes
    import torch
    from paper_1503_00757_gb300.binding import Context, Context3D, lib
    L = lib()
    mT, mR, v, vt = _inputs()
    rng = np.random.default_rng(6)
    m3 = [to_gpu(rng.random((16, 16, 16))) for _ in range(2)]
    v3, t3 = (to_gpu(0.1 * rng.standard_normal((3, 16, 16, 16))) for _ in range(2))
    E = lambda k: torch.zeros(k, N, N, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())

    def calls():
        s = torch.cuda.Stream() if working_stream else None
        ctx, c3 = Context(N, N, NT, stream=s), Context3D(16, 16, 16, 2, stream=s)
        u, det, m1, g, H, H3 = E(2), E(1), E(1), E(2), E(2), torch.zeros_like(v3)
        torch.cuda.synchronize()
        ctx.set_images(mT, mR)
        c3.set_images(*m3)
        c3.gradient(v3, H3)
        todo = [lambda: L.reg_displacement(ctx.h, p(v), p(u)), lambda: L.reg3_hessian_matvec(c3.h, p(t3), p(H3)),
                lambda: L.reg_detgrad(ctx.h, p(v), p(det), None), lambda: L.reg_objective(ctx.h, p(v), p(m1), None),
                lambda: L.reg_gradient(ctx.h, p(v), p(g), None), lambda: L.reg_hessian_matvec(ctx.h, p(vt), p(H))]
        # dropping captured sequences counts as well
        todo += [lambda: L.reg_set_params(ctx.h, NT, 1, 2e-2, math.inf, 0.0)]
        torch.cuda.synchronize()
        return ctx, c3, todo, (u, det, m1, g, H, H3)

    ctx, c3, todo, ref = calls()
    assert [f() for f in todo] == [0] * len(todo)
    torch.cuda.synchronize()
    ctx.close()
    c3.close()
    ctx, c3, todo, out = calls()
    x, other, graph = torch.zeros(4, device="cuda"), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=other):
        x.add_(1)
        rcs = [f() for f in todo]
        x.add_(1)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    ctx.close()
    c3.close()
    assert rcs == [0] * len(todo)
    assert bool((x == 2).all())
    assert all(torch.equal(a, b) for a, b in zip(ref, out))


@pytest.mark.parametrize("called_before", [False, True])
def test_refused_calls_leave_the_context_and_the_capture_as_they_were(called_before):
    """Objective, gradient, matvec and det F are refused on a stream that is being captured; the
    linearization point and the caller's graph do not notice."""
    import ctypes
    import torch
    from paper_1503_00757_gb300.binding import Context, lib
    L = lib()
    mT, mR, v, vt = _inputs()
    s = torch.cuda.Stream()
    ctx = Context(N, N, NT, stream=s)
    E = lambda k: torch.zeros(k, N, N, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    g, H, H2, w, x = E(2), E(2), E(2), (0.5 * v).contiguous(), torch.zeros(4, device="cuda")
    torch.cuda.synchronize()
    ctx.set_images(mT, mR)
    if called_before:
        ctx.detgrad(v)
        ctx.objective(v)
    ctx.gradient(v, g)
    ctx.hessian_matvec(vt, H)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        x.add_(1)
        rcs = [L.reg_gradient(ctx.h, p(w), p(g), None), L.reg_objective(ctx.h, p(w), None, None),
               L.reg_hessian_matvec(ctx.h, p(w), p(H)), L.reg_detgrad(ctx.h, p(w), None, None)]
        x.add_(1)
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert rcs == [2, 2, 2, 2]  # REG_ERR_CUDA
    assert bool((x == 2).all())
    ctx.hessian_matvec(vt, H2)
    torch.cuda.synchronize()
    ctx.close()
    assert torch.equal(H, H2)


@pytest.mark.parametrize("working_stream", [False, True])
def test_first_calls_while_another_thread_synchronizes_the_device(working_stream):
    """While a stream is being captured no thread may synchronize the device: a context's first calls
    capture nothing, so neither side of this fails, and the results are the usual ones."""
    import threading
    import torch
    from paper_1503_00757_gb300.binding import Context, Context3D
    mT, mR, v, vt = _inputs()
    rng = np.random.default_rng(6)
    m3 = [to_gpu(rng.random((16, 16, 16))) for _ in range(2)]
    v3, t3 = (to_gpu(0.1 * rng.standard_normal((3, 16, 16, 16))) for _ in range(2))
    s = torch.cuda.Stream() if working_stream else None
    torch.cuda.synchronize()

    def once():
        E = lambda k: torch.zeros(k, N, N, device="cuda")
        out = g, H, u, det, v1, H3 = E(2), E(2), E(2), E(1), E(2), torch.zeros_like(v3)
        ctx, c3 = Context(N, N, NT, regnorm=2, beta=1e-2, stream=s), Context3D(16, 16, 16, 2, stream=s)
        ctx.set_images(mT, mR)
        c3.set_images(*m3)
        for _ in range(12):
            ctx.displacement(v, u)
            ctx.gradient(v, g)
            ctx.hessian_matvec(vt, H)
        ctx.detgrad(v, det)
        c3.gradient(v3, H3)
        c3.hessian_matvec(t3, H3)
        from paper_1503_00757_gb300.binding import default_opts
        ctx.solve(v1, default_opts(maxit_newton=1, maxit_pcg=3), check=False)
        torch.cuda.synchronize()
        ctx.close()
        c3.close()
        return out

    ref = once()
    stop, failed, count = threading.Event(), [], [0]

    def other():
        while not stop.is_set():
            try:
                torch.cuda.synchronize()
                count[0] += 1
            except Exception as e:  # noqa: BLE001
                failed.append(str(e))

    t = threading.Thread(target=other)
    t.start()
    try:
        outs = [once() for _ in range(12)]
    finally:
        stop.set()
        t.join()
    assert not failed and count[0] > 0
    for o in outs:
        assert all(torch.equal(a, b) for a, b in zip(o, ref))
