"""The TMA-fed convolution (opnet_conv / opnet_conv_dgrad on the tensor cores, input channels a
multiple of 8) on small integers: BF16 holds the operands and FP32 every partial sum exactly, so
the result must equal the integer convolution bit for bit.  Channel counts cover every split of
a tap into pieces of 64, 32, 16 and straddling 8 + 8 values, and K ending on half a step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402


def conv_int(X, N, taps, W):
    """sum_t X[m + off_t] W[t] in int64, zero outside the grid."""
    cin = X.shape[1]
    if taps == 1:
        return X @ W
    P = np.zeros((N + 2, N + 2, N + 2, cin), dtype=np.int64)
    P[1:-1, 1:-1, 1:-1] = X.reshape(N, N, N, cin)
    out = np.zeros((N**3, W.shape[1]), dtype=np.int64)
    for t in range(27):
        z, y, x = t // 9, t // 3 % 3, t % 3
        out += P[z:z + N, y:y + N, x:x + N].reshape(-1, cin) @ W[t * cin:(t + 1) * cin]
    return out


@pytest.mark.parametrize("cin", [3, 4, 6, 9, 12, 8, 16, 24, 32, 40, 48, 56, 72, 96, 104, 144, 200])
@pytest.mark.parametrize("N,taps,cout", [(1, 27, 8), (4, 27, 24), (5, 27, 128), (7, 27, 50), (12, 27, 48),
                                         (5, 1, 64), (6, 1, 3)])
def test_conv_is_exact_on_integers(cin, N, taps, cout):
    rng = np.random.default_rng(cin * N + taps + cout)
    X = rng.integers(-8, 9, (N**3, cin))
    W = rng.integers(-4, 5, (taps * cin, cout))
    b = rng.integers(-9, 10, cout)
    dev = lambda a: torch.from_numpy(a.astype(np.float32)).cuda()  # noqa: E731
    Z, A = pkg.binding.net_conv("bf16_tc", dev(X), N, taps, dev(W), dev(b))
    want = conv_int(X, N, taps, W) + b
    got = Z.cpu().numpy()
    assert np.array_equal(got, want.astype(np.float32))
    z = want.astype(np.float64)
    silu = z / (1.0 + np.exp(np.minimum(-z, 700.0)))
    assert np.all(np.abs(A.cpu().numpy() - silu) <= 1e-6 * np.abs(silu) + 1e-30)
    if cout % 8 == 0 and cin <= 128:  # the adjoint: the same kernel on cout input channels
        dZ = rng.integers(-8, 9, (N**3, cout))
        dX = pkg.binding.net_conv_dgrad("bf16_tc", dev(dZ), N, taps, dev(W)).cpu().numpy()
        Wf = np.concatenate([W[t * cin:(t + 1) * cin].T for t in range(taps - 1, -1, -1)])
        assert np.array_equal(dX, conv_int(dZ, N, taps, Wf).astype(np.float32))
