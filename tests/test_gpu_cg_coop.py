"""Step 1 in one cooperative launch (op_cg_solve on blocks that stay in L2): one CTA, one
cluster, a grid of CTAs with a ragged last one, at the sizes where the split changes.

Every column must meet ||u - (H + sigma) w|| <= rtol ||u||, checked in FP64 with the oracle's H
on the rounded inputs.  CG stops on its recursive residual, which drifts from the true one by
a few roundings of (H + sigma) w per iteration: with ||H + sigma|| ||w|| <= kappa ||u||, the
tolerance adds iterations * eps * kappa."""
import numpy as np
import pytest
import scipy.sparse

import oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402

# (shape, p): 1 point; a thread block's points and one more; a cluster's range and one past it
# (ld 8 FP32: 256 rows a CTA, FP64: 128); a full grid; wide rows; odd axes
SIZES = [((1, 1), 1), ((16, 16), 8), ((257, 1), 7), ((128, 128), 8), ((127, 129), 8), ((128, 129), 3),
         ((16, 8, 128), 8), ((7, 5, 3), 60), ((33, 31, 29), 61), ((21, 20, 19), 129), ((9, 8, 7), 250)]


@pytest.mark.parametrize("shape,p", SIZES, ids=[f"{'x'.join(map(str, s))}_p{p}" for s, p in SIZES])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64], ids=["fp32", "fp64"])
@pytest.mark.parametrize("precond", ["none", "jacobi"])
def test_solution_meets_the_residual_test(shape, p, dtype, precond):
    n, ld = int(np.prod(shape)), (p + 7) // 8 * 8
    p = min(p, n)
    rng = np.random.default_rng(n + p)
    lo, hi = (-1.0,) * len(shape), (1.0,) * len(shape)
    np_t = np.float32 if dtype == torch.float32 else np.float64
    V = (20.0 * rng.random(n)).astype(np_t)
    U = np.zeros((n, ld), dtype=np_t)
    U[:, :p] = rng.standard_normal((n, p))
    W0 = np.zeros_like(U)
    W0[:, :p] = 0.01 * rng.standard_normal((n, p))  # a warm start
    if p > 2:
        U[:, 1] = 0.0  # a zero column is left alone
        W0[:, 1] = 0.0
    rtol, eps = (1e-4, 2.0**-23) if dtype == torch.float32 else (1e-10, 2.0**-52)
    Ud, Wd = torch.from_numpy(U).cuda(), torch.from_numpy(W0).cuda()
    its = pkg.cg_solve(shape, lo, hi, torch.from_numpy(V).cuda(), 1.0, Ud, Wd, p, rtol, precond=precond)
    W = Wd.cpu().numpy().astype(np.float64)
    H = o.hamiltonian(shape, lo, hi, V.astype(np.float64))
    A = H + scipy.sparse.identity(n)
    res = np.linalg.norm(U.astype(np.float64) - A @ W, axis=0)
    # ||H + sigma|| <= largest row sum; (H + sigma)^-1 <= 1
    kappa = float(abs(A).sum(axis=1).max())
    tol = (rtol + 2 * (its + 1) * eps * kappa) * np.linalg.norm(U.astype(np.float64), axis=0)
    assert np.all(res <= tol), float((res / np.maximum(tol, 1e-300)).max())
    assert np.all(W[:, p:] == 0.0)
    if p > 2:
        assert np.all(W[:, 1] == 0.0)
    # the same call again: the same bits, and no iteration from a converged start
    Wd2 = torch.from_numpy(W0).cuda()
    assert pkg.cg_solve(shape, lo, hi, torch.from_numpy(V).cuda(), 1.0, Ud, Wd2, p, rtol, precond=precond) == its
    assert torch.equal(Wd, Wd2)
    capped = torch.from_numpy(W0).cuda()
    assert pkg.cg_solve(shape, lo, hi, torch.from_numpy(V).cuda(), 1.0, Ud, capped, p, 0.0, max_iter=3,
                        precond=precond) <= 3
