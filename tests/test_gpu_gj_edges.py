"""The FP32 seed of the Step-2 inverse at block widths around its groups of 8 pivots, its 32-row
warps and its 128-column limit.

A batch has no fallback behind the seed (a single solve replaces a bad inverse by the LU one), so a
wrong seed shows there: the steps must keep <U, U> = I and agree with the single solves.  Bound on
|<U, U> - I|_F: every step rounds p x p coefficients to FP32 and sums 2 p products with 2^-20
relative error each, 5 steps of 2^-20 p in all; the energies differ by the rounding of differently
partitioned sums, 2e-5 as in the other batch tests."""
import numpy as np
import pytest

import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402

WIDTHS = [1, 7, 8, 9, 24, 31, 33, 64, 100, 121, 127, 128]


def test_steps_keep_orthonormality_at_every_width():
    probs = [syn.wells_3d(9, p, 4, p) for p in WIDTHS]

    def solvers():
        return [pkg.Solver(P.shape, P.lo, P.hi, P.V, syn.gaussian_block(i, P.n, P.p), P.p, prec="fp32")
                for i, P in enumerate(probs)]

    single, batched = solvers(), solvers()
    for s in single:
        s.step(5)
    with pkg.Batch(batched, cg_iters=200) as b:
        b.step(5)
        for s1, s2, P in zip(single, batched, probs):
            assert s2.stats()["energy"] == pytest.approx(s1.stats()["energy"], rel=2e-5)
            U = s2.get_U().astype(np.float64)
            assert np.linalg.norm(U.T @ U - np.eye(P.p)) <= 5 * 2.0**-20 * P.p + 1e-6, P.p
    for s in single + batched:
        s.close()
