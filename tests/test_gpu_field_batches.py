"""The transforms have kernels for one field, for many equally spaced ones (which also scale) and for
two (csrc/kernels.cu, Fields): a batch gives what its members give alone, on a grid of one row tile
and on larger ones, and a scaled result is the scaled unscaled one (one rounding, so bit for bit)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("H,W", [(32, 32), (32, 128), (128, 64)])
def test_output_map_of_a_batch_equals_its_members(H, W):
    import torch
    from paper_1503_00757_gb300.binding import Net
    rng = np.random.default_rng(H + W)
    net = Net(H, W, 3)
    p = torch.tensor(0.1 * rng.standard_normal(net.nparams), dtype=torch.float32, device="cuda")
    images = torch.tensor(rng.random((3, 2, H, W)), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    net.set_params(p)
    out, one = torch.empty(3, 2, H, W, device="cuda"), torch.empty(3, 2, H, W, device="cuda")
    net.forward(images, out)
    for b in range(3):
        net.forward(images[b:b + 1], one[b:b + 1])
    assert torch.equal(out, one)
    net.set_output_scale(0.3)
    scaled, scaled_one = torch.empty_like(out), torch.empty_like(out)
    net.forward(images, scaled)
    for b in range(3):
        net.forward(images[b:b + 1], scaled_one[b:b + 1])
    torch.cuda.synchronize()
    net.close()
    assert torch.equal(scaled, out * torch.tensor(0.3, dtype=torch.float32, device="cuda"))
    assert torch.equal(scaled, scaled_one)


def test_fine_warm_start_refuses_a_misaligned_output():
    import ctypes
    import torch
    from paper_1503_00757_gb300.binding import Net, lib
    net = Net(32, 32, 1)
    images, buf = torch.rand(1, 2, 64, 64, device="cuda"), torch.zeros(2 * 64 * 64 + 4, device="cuda")
    torch.cuda.synchronize()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert lib().reg_net_forward_fine(net.h, p(images), 1, p(buf[1:])) == 1  # REG_ERR_ARG
    assert b"16-byte aligned" in lib().reg_last_error()
    assert lib().reg_net_forward_fine(net.h, p(images), 1, p(buf)) == 0
    torch.cuda.synchronize()
    net.close()
