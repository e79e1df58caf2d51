"""The row form of the compact right side (one warp per x row, the terms of a row 32 at a time)
against the oracle's assembly: at, below and above a pass of 32 terms, rows shorter and longer
than a warp, every face kind on every axis, Gaussian tails that underflow to zero, and complex
separable factors."""
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


@pytest.mark.parametrize("n,nsrc,k,faces", [
    (3, 1, 2.0, "NNNNNN"), (30, 31, 7.0 + 0.3j, "DNNDSS"), (31, 32, 9.0, "SSDNND"), (33, 33, 11.0, "NDSDNN"),
    (90, 70, 20.0 + 0.2j, "NNDDNS"), (96, 2, 25.0, "DDNNSS")])
def test_gaussian_rows(H, n, nsrc, k, faces):
    src = inputs.gaussian_sources(5 + n, n, nsrc, margin_h=1)
    prob = O.Problem(n, k, faces)
    with H.Solver(n, k, faces, method=H.SKS) as s:
        F = s.rhs_gaussians(src).cpu().numpy()
    ref = O.rhs(prob, O.sources.gaussians(src))
    # at most a few dozen roundings per term, of terms no larger than the field's maximum times
    # the table values' own error (the Gaussian's argument): 1e-12 of the maximum
    assert np.abs(F - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("nt", [1, 33])
def test_complex_rows(H, nt):
    """A sum of separable terms equals the sum of the terms assembled one at a time."""
    n, faces = 20, "NNDNSS"
    rng = np.random.default_rng(7)
    with H.Solver(n, 6.0, faces, method=H.SKS) as s:
        m = max(s.dims)
        tab = rng.standard_normal((nt, 3, 5, m)) + 1j * rng.standard_normal((nt, 3, 5, m))
        cf = rng.standard_normal(nt) + 1j * rng.standard_normal(nt)
        F = s.rhs_separable(cf, tab).cpu().numpy()
        ref = sum(s.rhs_separable(cf[t:t + 1], tab[t:t + 1]).cpu().numpy() for t in range(nt))
    assert np.isfinite(F).all() and np.abs(F - ref).max() <= 1e-13 * np.abs(ref).max()
