"""Grids whose stencil blocks hold fewer planes than a full chunk (the planes per block follow the
number of blocks), in both precisions: the operator against the oracle at plane counts around the
chunk lengths 2, 4, 8, 16 and the tiles of 32 points."""
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


@pytest.mark.parametrize("n,faces", [(1, "NNNNSS"), (2, "DDNNSS"), (3, "DNDNDS"), (16, "NNDDSD"), (31, "DDNNSS"),
                                     (33, "NDDNNN"), (64, "DDNNSS"), (95, "DDDDNS"), (127, "DDNNSS")])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("mixed", 4e-6)])
def test_operator_small_chunks(H, n, faces, precision, tol):
    prob = O.Problem(n, 0.2 * (n + 1) + 0.1j, faces)
    x = inputs.complex_normal(n, prob.shape)
    ref = O.apply_A(prob, x)
    with H.Solver(n, prob.k, faces, precision=H.FP64 if precision == "fp64" else H.MIXED, method=H.SKS) as s:
        y = s.apply_A(torch.from_numpy(x).cuda()).cpu().numpy()
    # 27 roundings of terms of the field's size: FP64 27 2^-53, FP32 27 2^-24 with the inputs' own
    assert np.abs(y - ref).max() <= tol * np.abs(ref).max()
