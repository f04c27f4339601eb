"""The FP32 inner matrices on the tensor cores at the edges of slabs (32 points), chunks (512),
tiles (128 columns) and of the persistent grid, for every subset of the products, against the
FP64 product.  Bound per entry: TF32 split 2^-21, 16 truncated MMAs a slab (16 2^-23), up to
64 slabs of a chunk added in FP32 (64 2^-24), partials added exactly: below 2^-17 sum |a| |b|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("p", [1, 20, 128, 130, 264])
@pytest.mark.parametrize("n", [1, 31, 33, 511, 513, 5000, 70001])
@pytest.mark.parametrize("want", [("C", "S", "D"), ("D",), ("C",)], ids=["CSD", "D", "C"])
def test_gram_of_ragged_blocks(n, p, want):
    rng = np.random.default_rng(n + p)
    ld = (p + 7) // 8 * 8
    U, W = (np.zeros((n, ld), dtype=np.float32) for _ in range(2))
    U[:, :p], W[:, :p] = rng.standard_normal((n, p)), rng.standard_normal((n, p))
    Ud, Wd = torch.from_numpy(U).cuda(), torch.from_numpy(W).cuda()
    got = dict(zip("CSD", pkg.gram(Ud, Wd, p, want=want)))
    again = dict(zip("CSD", pkg.gram(Ud, Wd, p, want=want)))
    U, W = U.astype(np.float64), W.astype(np.float64)
    for k, (A, B) in {"C": (W, U), "S": (W, W), "D": (U, U)}.items():
        if k not in want:
            assert got[k] is None
            continue
        g = got[k].cpu().numpy()
        bound = 2.0**-17 * (np.abs(A).T @ np.abs(B)) + 1e-30
        err = np.abs(g - A.T @ B)
        assert np.all(err <= bound), (k, float((err / bound).max()))
        assert torch.equal(got[k], again[k])  # a fixed order of sums
        if k != "C":  # the tiles below the diagonal are copies (a diagonal tile rounds each side)
            assert np.array_equal(g[:128, 128:], g[128:, :128].T)
