"""Step 1 of FP32 blocks whose column sums leave the FP32 range while every element, product and
point stays inside it: |u_i| up to 1.5e18, so u_i^2 < 2.3e36 and ||u||^2 is 2e38 .. 2e41.

Every column, large and ordinary, must meet ||u - (H + sigma) w|| <= rtol ||u|| as in
tests/test_gpu_cg_coop.py (its tolerance: rtol plus two roundings of (H + sigma) w an iteration).
One CTA, one cluster, a grid of CTAs, and blocks of the general kernels (ld > 256)."""
import numpy as np
import pytest
import scipy.sparse

import oracle as o

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("shape,p", [((16, 16), 8), ((128, 128), 8), ((150, 151), 5), ((31, 30, 29), 40),
                                     ((9, 8, 7), 260)], ids=lambda v: str(v).replace(" ", ""))
@pytest.mark.parametrize("precond", ["none", "jacobi"])
def test_columns_of_large_norm_are_solved(shape, p, precond):
    n, ld = int(np.prod(shape)), (p + 7) // 8 * 8
    rng = np.random.default_rng(n)
    half = 0.25 * max(shape)  # a mesh width near 1/2
    lo, hi = (-half,) * len(shape), (half,) * len(shape)
    V = (4.0 * rng.random(n)).astype(np.float32)
    U = np.zeros((n, ld), np.float32)
    U[:, :p] = rng.uniform(-1.0, 1.0, (n, p))
    U[:, 0:p:2] *= np.float32(1.5e18)
    U[:, 1] *= np.float32(1e-12)
    Ud, Wd = torch.from_numpy(U).cuda(), torch.zeros(n, ld, device="cuda")
    rtol, eps = 1e-4, 2.0**-23
    its = pkg.cg_solve(shape, lo, hi, torch.from_numpy(V).cuda(), 1.0, Ud, Wd, p, rtol, precond=precond)
    assert its > 0
    A = o.hamiltonian(shape, lo, hi, V.astype(np.float64)) + scipy.sparse.identity(n)
    kappa = float(abs(A).sum(axis=1).max())
    W, U = Wd.cpu().numpy().astype(np.float64), U.astype(np.float64)
    norm = np.linalg.norm(U, axis=0)
    assert np.any(np.sum(U * (A @ U), axis=0) > 3.4e38)  # (P . A P of the first iteration, unpreconditioned)
    res = np.linalg.norm(U - A @ W, axis=0)
    tol = (rtol + 2 * (its + 1) * eps * kappa) * norm
    assert np.all(res <= tol), float((res[:p] / tol[:p]).max())


@pytest.mark.parametrize("shape,p", [((16, 16), 8), ((128, 128), 8), ((31, 30, 29), 40)],
                         ids=lambda v: str(v).replace(" ", ""))
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64], ids=["fp32", "fp64"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_column_leaves_the_others_alone(shape, p, dtype, bad):
    """Cooperative solve and general kernels: the other columns meet the residual test, and the solve
    ends with them (a NaN column is inactive from the start, an infinite one has no finite target)."""
    n = int(np.prod(shape))
    rng = np.random.default_rng(n + 1)
    half = 0.25 * max(shape)
    lo, hi = (-half,) * len(shape), (half,) * len(shape)
    np_t = np.float32 if dtype == torch.float32 else np.float64
    V = (4.0 * rng.random(n)).astype(np_t)
    U = rng.uniform(-1.0, 1.0, (n, p)).astype(np_t)
    U[n // 3, 2] = bad
    rtol, eps = (1e-4, 2.0**-23) if dtype == torch.float32 else (1e-10, 2.0**-52)
    A = o.hamiltonian(shape, lo, hi, V.astype(np.float64)) + scipy.sparse.identity(n)
    kappa = float(abs(A).sum(axis=1).max())
    keep = np.arange(p) != 2
    Vd, Ud = torch.from_numpy(V).cuda(), torch.from_numpy(U).cuda()
    for route in (0, 1):
        Wd = torch.zeros_like(Ud)
        args = (shape, lo, hi, Vd, 1.0, Ud, Wd, p, rtol)
        its = pkg.cg_solve(*args) if route == 0 else pkg.selftest_cg(route, *args)
        assert 0 < its < 500
        W, Uk = Wd.cpu().numpy().astype(np.float64)[:, keep], U.astype(np.float64)[:, keep]
        res = np.linalg.norm(Uk - A @ W, axis=0)
        assert np.all(res <= (rtol + 2 * (its + 1) * eps * kappa) * np.linalg.norm(Uk, axis=0)), route
