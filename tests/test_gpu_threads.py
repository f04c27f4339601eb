"""Host threads, each with its own stream, in calls that share a kernel but ask for different
amounts of shared memory: every call succeeds and returns the bits it returns alone.  (The
cooperative solve in a cluster of CTAs takes about 75 KB at ld = 64 and 56 KB at ld = 40, the
convolutions and weight gradients differ by their channels.)  A refused
cooperative launch shows in the bits: the solve then takes the general path."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402
from tests.test_gpu_opnet import DEV, GAMMA, setup, target  # noqa: E402


def steps(shape, p, seed):
    n = int(np.prod(shape))
    rng = np.random.default_rng(seed)
    V, U0 = rng.random(n), rng.standard_normal((n, p))

    def call():
        with pkg.Solver(shape, (-1.0,) * 3, (1.0,) * 3, V, U0, p, prec="fp32", cg_rtol=0.3) as s:
            s.step(500)
            return s.get_U_device(torch.float32)
    return call


def conv(N, cin, cout, seed):
    rng = np.random.default_rng(seed)
    X = torch.from_numpy(rng.standard_normal((N**3, cin)).astype(np.float32)).to(DEV)
    W = torch.from_numpy(rng.standard_normal((27 * cin, cout)).astype(np.float32)).to(DEV)
    return lambda: pkg.binding.net_conv("bf16_tc", X, N, 27, W)[0]


def gradient(widths, seed):
    net, _, P, V = setup(8, widths, 8, seed=seed)
    Us = torch.from_numpy(target(P.n, 8, 5)).to(DEV, torch.float32)
    return lambda: torch.from_numpy(net.loss_grad(V, Us, GAMMA)[1])


@pytest.mark.parametrize("make,calls", [
    (lambda: (steps((8, 8, 8), 64, 1), steps((8, 8, 8), 40, 2)), 10),
    (lambda: (conv(6, 8, 16, 3), conv(6, 128, 128, 4)), 3000),
    (lambda: (gradient((4, 4, 4), 5), gradient((64, 64, 64), 6)), 300)],
    ids=["cg", "conv", "weight_gradient"])
def test_threads_with_different_shared_memory(make, calls):
    jobs = make()
    want = [job() for job in jobs]
    torch.cuda.synchronize()
    failed = []

    def work(i):
        stream = torch.cuda.Stream()
        try:
            with torch.cuda.stream(stream):
                for _ in range(calls):
                    if not torch.equal(jobs[i](), want[i]):
                        failed.append((i, "other bits"))
                        return
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            failed.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
