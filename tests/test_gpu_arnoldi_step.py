"""The Arnoldi step's small algebra (column sums, rotations kept as their product, triangular
solves spread over lanes) at restart lengths around its rows of 32 lanes and eight warps: GMRES and
flexible GMRES in FP64 against the oracle's GMRES of the same restart length."""
import numpy as np
import pytest

import helm6_inputs as inputs
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1212_1397_gb300 import build, helm6
    build.build()
    return helm6


@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 31, 32, 33, 64])
@pytest.mark.parametrize("method", ["gmres", "fgmres"])
def test_estimate_is_the_residual(H, m, method):
    """The residual estimate of the last column (rotations, recurrences) is the true residual of the
    iterate the least-squares solution gives, on a problem that no cycle of these lengths solves."""
    n, k, faces = 16, 26.0 + 0.3j, "DDNNDD"
    prob = O.Problem(n, k, faces)
    F = inputs.complex_normal(m, prob.shape)
    meth = {"gmres": H.GMRES, "fgmres": H.FGMRES}[method]
    with H.Solver(n, k, faces, precision=H.FP64, method=meth, max_restart=64) as s:
        u, st = s.solve(torch.from_numpy(F).cuda(), tol=1e-12, restart=m, maxit=m)
    res = np.linalg.norm(F - O.apply_A(prob, u.cpu().numpy())) / np.linalg.norm(F)
    assert st["iters"] == m and res < 1.0
    # both are the norm of the same vector; the Arnoldi relation holds to a few 2^-53 of ||A M^-1|| (some
    # tens here) over residuals above 1e-6
    assert abs(st["relres"] - res) <= 1e-7 * res and abs(st["history"][-1] - res) <= 1e-7 * res, (st["history"][-1], res)


@pytest.mark.parametrize("m", [1, 2, 8, 9, 32, 64])
def test_counts(H, m):
    """An easy problem: the oracle's iteration count (within one) and solution at every restart length."""
    n, k, faces, tol = 16, 11.0 + 0.6j, "DDNNDD", 1e-10
    prob = O.Problem(n, k, faces)
    F = inputs.complex_normal(m, prob.shape)
    U, info = O.gmres(lambda v: O.apply_A(prob, v), O.Preconditioner(prob), F, tol=tol, restart=m, maxit=400)
    with H.Solver(n, k, faces, precision=H.FP64, max_restart=64) as s:
        u, st = s.solve(torch.from_numpy(F).cuda(), tol=tol, restart=m, maxit=400)
    assert st["rc"] == 0 and abs(st["iters"] - info["iters"]) <= 1, (st["iters"], info["iters"])
    # two iterates with residuals of 1e-10: their distance is that times ||A^-1|| ||F|| / ||U||, some tens
    assert np.linalg.norm(u.cpu().numpy() - U) <= 1e-7 * np.linalg.norm(U)
