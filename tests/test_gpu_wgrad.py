"""The weight gradients of the warm-start network over the shapes that change their launch:
one, three or nine (dz, dy) groups a CTA, several k blocks, one or many point runs, channels
that are multiples of 4 but not of 8, and the gathered form for the others; FP32 convolutions,
against the oracle's gradient with the tolerance of tests/test_gpu_opnet.py (1e-4 per layer)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

from oracle import unet  # noqa: E402
from tests.test_gpu_opnet import DEV, GAMMA, layer_slices, setup, target  # noqa: E402


@pytest.mark.parametrize("N,widths,p", [(4, (24, 48, 96), 8), (12, (24, 48, 96), 64), (8, (128, 128, 128), 8),
                                        (8, (4, 12, 20), 16), (8, (8, 100, 4), 8), (16, (16, 8, 8), 8),
                                        (8, (24, 6, 96), 8)])
def test_weight_gradients_match_oracle(N, widths, p):
    net, theta, P, V = setup(N, widths, p, seed=7)
    net.set_conv("fp32")
    Us = target(P.n, p, 5)
    loss, g = net.loss_grad(V, torch.from_numpy(Us).to(DEV, torch.float32), GAMMA)
    Y_ref, cache = unet.forward(theta, P.V, N, P.lo, P.hi, widths, p)
    ref_loss, dY = unet.subspace_loss(Y_ref, Us, GAMMA)
    g_ref = unet.backward(cache, dY)
    assert abs(loss - ref_loss) <= 2e-5 * abs(ref_loss)
    table = unet.layer_table(*widths, p)
    for (name, *_), sl in zip(table, layer_slices(table)):
        err = np.linalg.norm(g[sl] - g_ref[sl]) / np.linalg.norm(g_ref[sl])
        assert err < 1e-4, (name, err)
    net.close()
