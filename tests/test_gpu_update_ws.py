"""The FP32 update on the tensor cores for block widths that are not multiples of the 32-column
slabs or the 128-column tiles, and ragged point counts, against the FP64 product.

Bound per entry: the TF32 split keeps products to 2^-22, a slab adds 12 truncated MMAs
(12 2^-23), the slabs are added in FP32: in all below 2^-19 sum |a| |b|, plus one rounding of
U + correction."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("p", [1, 8, 20, 40, 64, 84, 100, 128, 136, 200, 264])
@pytest.mark.parametrize("n", [1, 127, 129, 20011])
def test_update_of_ragged_blocks(n, p):
    rng = np.random.default_rng(n + p)
    ld = (p + 7) // 8 * 8
    U, W = (rng.standard_normal((n, p)).astype(np.float32) for _ in range(2))
    KU = (np.eye(p) + 0.1 * rng.standard_normal((p, p))).astype(np.float32)
    KW = (0.5 * rng.standard_normal((p, p))).astype(np.float32)

    def pad(A, rows):
        out = torch.zeros(rows, ld, device="cuda")
        out[: A.shape[0], : A.shape[1]] = torch.from_numpy(A).cuda()
        return out

    got = pkg.update(pad(U, n), pad(W, n), pad(KU, ld), pad(KW, ld), p).cpu().numpy().astype(np.float64)
    assert np.all(got[:, p:] == 0.0)
    U, W, KU, KW = (A.astype(np.float64) for A in (U, W, KU, KW))
    D = KU - np.eye(p)
    want = U + U @ D + W @ KW
    bound = 2.0**-19 * (np.abs(U) @ np.abs(D) + np.abs(W) @ np.abs(KW)) + 2.0**-22 * np.abs(want) + 1e-30
    err = np.abs(got[:, :p] - want)
    assert np.all(err <= bound), float((err / bound).max())
