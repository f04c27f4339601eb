"""The digit splitting and the integer epilogue of the FP64 tensor-core update at the edges of
their ranges: products with powers of two, where the result is exact (or one rounding of an
exact value at the ends of the FP64 range), so every comparison is bitwise."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402


def edge_values(n, p, seed):
    """53-bit values of both signs within a factor of 256 of the largest of their row."""
    rng = np.random.default_rng(seed)
    m = rng.integers(2**52, 2**53, (n, p), dtype=np.int64)
    special = np.array([2**53 - 1, 2**52, 2**52 + 1, 0x10808080808080, 0x1F7F7F7F7F7F7F, 0x18000000000000,
                        0x17FFFFFFFFFFFF, 0x10000000000080, 0x1000000000007F], dtype=np.int64)
    pick = rng.random((n, p)) < 0.5
    m = np.where(pick, special[rng.integers(0, len(special), (n, p))], m)
    x = np.ldexp(m.astype(np.float64), rng.integers(-60, -52, (n, p)))
    x[rng.random((n, p)) < 0.05] = 0.0
    return np.where(rng.random((n, p)) < 0.5, x, -x)


@pytest.mark.parametrize("n,p", [(1, 8), (129, 8), (130, 72), (257, 200)])
@pytest.mark.parametrize("scale", [-900, 0, 900])
def test_negation_is_exact(n, p, scale):
    U = np.ldexp(edge_values(n, p, n + p), scale)
    Ud = torch.from_numpy(U).cuda()
    KU = -torch.eye(p, dtype=torch.float64, device="cuda")
    got = pkg.binding.update_fp64tc(Ud, None, KU, None, p).cpu().numpy()
    assert np.array_equal(got, -U)


@pytest.mark.parametrize("scale,shift", [(-1005, -30), (-1000, -20), (1000, 30), (900, 20), (0, 0)])
def test_results_at_the_ends_of_the_range_round_once(scale, shift):
    n, p = 131, 16
    W = np.ldexp(edge_values(n, p, 7), scale)
    U = np.zeros_like(W)
    eye = torch.eye(p, dtype=torch.float64, device="cuda")
    got = pkg.binding.update_fp64tc(torch.from_numpy(U).cuda(), torch.from_numpy(W).cuda(), eye,
                                    eye * 2.0**shift, p).cpu().numpy()
    with np.errstate(over="ignore"):
        want = np.ldexp(W, shift)
    assert np.array_equal(got, want)
