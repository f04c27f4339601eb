"""FP32 inner matrices whose entries leave the FP32 range while every chunk's partial stays inside it:
|x| up to 2e17, so 512 points make at most 2.1e37 and 70001 points up to 2.8e39.  The entries are FP64
and keep the accuracy of tests/test_gpu_gram_ws.py (2^-17 sum |a| |b|; three BF16 pieces keep 2^-16
sum |a| |b|: 2^-24 each of six dropped products and the same FP32 sums).  A column that holds an
infinity spoils its own row and column only."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("prec,bits", [(None, 17), ("mix_bf16x3", 16)], ids=["fp32", "bf16x3"])
@pytest.mark.parametrize("p", [8, 136])
def test_entries_beyond_the_fp32_range(p, prec, bits):
    n = 70001
    rng = np.random.default_rng(p)
    U, W = (rng.uniform(-1.0, 1.0, (n, p)).astype(np.float32) for _ in range(2))
    U[:, ::3] *= np.float32(2e17)
    W[:, 1::3] *= np.float32(2e17)
    bad = p - 1
    U[n // 2, bad] = np.inf
    got = pkg.gram(torch.from_numpy(U).cuda(), torch.from_numpy(W).cuda(), p, prec=prec)
    C, S, D = (x.cpu().numpy() for x in got)
    assert not np.isfinite(D[bad]).any() and not np.isfinite(C[:, bad]).any()
    U[n // 2, bad] = 0.0
    keep = np.arange(p) != bad
    U, W = U.astype(np.float64), W.astype(np.float64)
    for name, g, A, B in (("C", C, W, U), ("S", S, W, W), ("D", D, U, U)):
        want, bound = A.T @ B, 2.0**-bits * (np.abs(A).T @ np.abs(B))
        cols = keep if name != "S" else np.ones(p, bool)
        rows = keep if name == "D" else np.ones(p, bool)
        err = np.abs(g - want)[np.ix_(rows, cols)]
        assert np.all(err <= bound[np.ix_(rows, cols)]), (name, err.max())
    assert np.abs(np.diag(S)).max() > 3.4e38
