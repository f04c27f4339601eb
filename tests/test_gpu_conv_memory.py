"""Convolutions and networks where the device has no room for the BF16 copy of the input that the
TMA-fed kernel reads: the kernel without a copy runs instead, with the same bits.  A tensor holds all
but a few MB of the device's memory meanwhile; outputs come from blocks torch has cached."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402
from tests.test_gpu_opnet import DEV, GAMMA, setup, target  # noqa: E402

MB = 1 << 20


def hold_all_but(left):
    torch.cuda.synchronize()
    return torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device=DEV)


# the copies: 8 channels of 106^3 points (three taps of 8 side by side) 57 MB, 72 of 58^3 28 MB
@pytest.mark.parametrize("kind,N,cin,cout,data", [("bf16_tc", 104, 8, 8, False), ("bf16_tc", 104, 8, 8, True),
                                                  ("fp32", 104, 8, 8, True), ("bf16_tc", 56, 136, 72, True)],
                         ids=["forward", "data_gradient", "data_gradient_fp32", "data_gradient_wide"])
def test_layer_without_room_for_the_copy(kind, N, cin, cout, data):
    rng = np.random.default_rng(cin)
    X = torch.from_numpy(rng.standard_normal((N**3, cout if data else cin)).astype(np.float32)).to(DEV)
    W = torch.from_numpy(rng.standard_normal((27 * cin, cout)).astype(np.float32)).to(DEV)

    def call():
        if data:
            return pkg.binding.net_conv_dgrad(kind, X, N, 27, W)
        return pkg.binding.net_conv(kind, X, N, 27, W)[0]

    want = call()
    call()  # (its output's block stays cached)
    hold = hold_all_but(16 * MB)
    try:
        got = call()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(got, want)


def test_network_without_room_for_the_copy():
    N, widths, p = 48, (24, 48, 96), 8  # largest copy: 144 values of 50^3 points, 34 MB
    free = torch.cuda.mem_get_info()[0]
    net, theta, P, V = setup(N, widths, p, conv="bf16_tc")
    Us = torch.from_numpy(target(P.n, p, 5)).to(DEV, torch.float32)
    Y, (loss, grad) = net.forward(V), net.loss_grad(V, Us, GAMMA)
    net.forward(V)
    torch.cuda.synchronize()
    net.close()
    probe = pkg.Net(N, P.lo, P.hi, p, widths)
    torch.cuda.synchronize()
    with_copy = torch.cuda.mem_get_info()[0]
    probe.close()
    torch.cuda.synchronize()
    size = torch.cuda.mem_get_info()[0] - with_copy
    assert 34 * MB < size < free
    hold = hold_all_but(size - 16 * MB)
    try:
        small = pkg.Net(N, P.lo, P.hi, p, widths)
        small.set_conv("bf16_tc")
        small.set_params(theta)
        Y2, (loss2, grad2) = small.forward(V), small.loss_grad(V, Us, GAMMA)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(Y, Y2) and loss == loss2 and np.array_equal(grad, grad2)
    small.close()
