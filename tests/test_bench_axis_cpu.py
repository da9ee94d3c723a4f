"""bench.py's byte and flop models of the axis-wise matvec, recounted launch by launch."""
import importlib.util
import math
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bench():
    spec = importlib.util.spec_from_file_location("bench_mod", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def test_axis_models():
    bench = _bench()
    for n1, n2, nt in [(512, 512, 32), (128, 1024, 7)]:
        N = n1 * n2
        # fields read + written per node: column launches (input, output; the adjoint's factor), then the
        # row launches of stage 1 and stage 2 (incremental state: u_s, D, v (2), u_out, stored source;
        # u_s, u_j, D, v (2), u_out, grad m (2), v~ (2), source stored; adjoint: lam, D, v_2, l_out;
        # the same with lam_j, b read and written (4) and grad m (2))
        state = (2 + 6) + (2 + 11)
        adjoint = (3 + 4) + (3 + 11)
        m = bench.matvec_models(n1, n2, nt, 1.0, 6805.0, 75.0)
        assert m["axis_pass"]["bytes"] == 4 * N * nt * (state + adjoint)
        assert abs(m["axis_pass"]["frac_hbm"] - m["axis_pass"]["bytes"] / 1e-3 / 1e9 / 6805.0) <= 1e-12
        fft = lambda n: 5 * n * math.log2(n)
        per_stage = 2 * (n2 // 2) * fft(n1) + 2 * (n1 // 2) * fft(n2)
        assert abs(m["axis_flops"]["flop"] - 4 * nt * per_stage) <= 1e-9 * m["axis_flops"]["flop"]
        assert abs(m["axis_flops"]["frac_fp32"] - 4 * nt * per_stage / 1e-3 / 1e12 / 75.0) <= 1e-9
    assert bench.matvec_models(64, 64, 4, 1.0, 1.0, 0.0)["axis_flops"]["frac_fp32"] is None
