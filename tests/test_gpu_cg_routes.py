"""The general kernels of Step 1 (stencil_cg.cu, stencil_tma.cu) where a small block would take the
cooperative launch: ragged x/y tiles and column chunks of the TMA direction kernel, 2-D row kernels,
the three-kernel FP64 iteration, and the solve after a refused cooperative launch; then blocks
beyond the cooperative sizes, by the rule.

Iterates against the oracle's block CG with the tolerances of tests/test_gpu_parity.py (2e-5 of the
largest entry in FP32, 1e-12 in FP64); large blocks by ||u - (H + sigma) w|| <= rtol ||u|| plus two
roundings of (H + sigma) w an iteration, as in tests/test_gpu_cg_coop.py."""
import numpy as np
import pytest
import scipy.sparse

import oracle as o
import synthetic as syn

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2511_06788_gb300 as pkg  # noqa: E402
from tests.test_gpu_parity import DEV, DT, TMA_GEOMS, ld_of, padded, random_potential, rounded  # noqa: E402

FORMS = [("fp32", g) for g in TMA_GEOMS] + [("fp32", ((17, 15), 24)), ("fp32", ((33, 1), 5)),
                                            ("fp32", ((9, 10, 2), 40)), ("fp32", ((11, 7, 5), 20)),
                                            ("fp64", ((13, 9, 11), 40)), ("fp64", ((17, 15), 12))]
IDS = [f"{a}_{'x'.join(map(str, g[0]))}_p{g[1]}" for a, g in FORMS]


@pytest.mark.parametrize("prec,geom", FORMS, ids=IDS)
@pytest.mark.parametrize("precond", ["none", "jacobi"])
def test_general_iterates_match_oracle(prec, geom, precond):
    shape, p = geom
    lo, hi = (-4.0,) * len(shape), (4.0,) * len(shape)
    n, ld = int(np.prod(shape)), ld_of(p)
    V = rounded(random_potential(shape, lo, hi, 5), prec)
    sigma = o.default_sigma(shape, lo, hi, V)
    U = rounded(o.householder_orthonormalize(syn.gaussian_block(6, n, p)), prec)
    W0 = rounded(0.05 * syn.gaussian_block(7, n, p), prec)
    A = (o.hamiltonian(shape, lo, hi, V) + sigma * scipy.sparse.identity(n)).tocsr()
    Vt, Ut = torch.from_numpy(V).to(DEV, DT[prec]), padded(U, ld, DT[prec])
    cg = o.block_pcg_jacobi if precond == "jacobi" else o.block_cg
    tol = 2e-5 if prec == "fp32" else 1e-12
    for k in (1, 2, 5):
        W_ref, _ = cg(A, U, W0, rtol=0.0, max_iter=k)
        got = []
        for route in (1, 2):
            Wt = padded(W0, ld, DT[prec])
            assert pkg.selftest_cg(route, shape, lo, hi, Vt, sigma, Ut, Wt, p, 1e-30, max_iter=k,
                                   precond=precond) == k
            got.append(Wt)
        assert torch.equal(got[0], got[1])
        W = got[0].double().cpu().numpy()
        assert np.abs(W[:, :p] - W_ref).max() < tol * np.abs(W_ref).max(), k
        assert np.all(W[:, p:] == 0)


@pytest.mark.parametrize("prec,shape,p", [("fp32", (97, 80, 71), 23), ("fp32", (64, 65, 67), 84),
                                          ("fp32", (1100, 1000), 12), ("fp64", (97, 80, 71), 35),
                                          ("fp64", (64, 63, 62), 129)])
@pytest.mark.parametrize("precond", ["none", "jacobi"])
def test_large_blocks_meet_the_residual_test(prec, shape, p, precond):
    n, ld = int(np.prod(shape)), ld_of(p)
    g = torch.Generator(device=DEV).manual_seed(p)
    V = 20.0 * torch.rand(n, generator=g, device=DEV, dtype=DT[prec])
    U = torch.zeros(n, ld, device=DEV, dtype=DT[prec])
    U[:, :p] = torch.randn(n, p, generator=g, device=DEV, dtype=DT[prec])
    W = torch.zeros_like(U)
    half = 0.25 * max(shape)  # a mesh width near 1/2
    lo, hi = (-half,) * len(shape), (half,) * len(shape)
    rtol, eps = (1e-4, 2.0**-23) if prec == "fp32" else (1e-10, 2.0**-52)
    its = pkg.cg_solve(shape, lo, hi, V, 1.0, U, W, p, rtol, precond=precond)
    assert 0 < its < 200
    A = (o.hamiltonian(shape, lo, hi, V.double().cpu().numpy()) + scipy.sparse.identity(n)).tocsr()
    kappa = float(abs(A).sum(axis=1).max())
    Uh, Wh = U.double().cpu().numpy(), W.double().cpu().numpy()
    norm = np.linalg.norm(Uh, axis=0)
    res = np.linalg.norm(Uh - A @ Wh, axis=0)
    assert np.all(res <= (rtol + 2 * (its + 1) * eps * kappa) * norm)
    assert np.all(Wh[:, p:] == 0)


def test_a_cooperative_solve_is_a_group_of_its_own_in_the_profile():
    P = syn.config_2d_laplace()
    with pkg.Solver(P.shape, P.lo, P.hi, P.V, syn.gaussian_block(0, P.n, P.p), P.p, prec="fp32") as s:
        s.profile(True)
        s.step(3)
        prof = s.profile_read()
    assert prof["cg_solve"][1] == 3 and prof["cg_solve"][0] > 0.0
    assert prof["cg_apply"][1] == 0 and prof["cg_axpy"][1] == 0
