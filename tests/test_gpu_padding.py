"""Rows of the mixed path's intermediates are padded to a multiple of 4; what the padding holds must
not reach a result.  Contexts are made in device memory that was filled with NaN before."""
import numpy as np
import pytest

import helm6_inputs as inputs
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,faces", [(9, "DNNDDN"), (13, "DDNNSS"), (14, "DDNNSD"), (30, "NNNDSS")])
def test_padding_is_not_read(n, faces):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1212_1397_gb300 import build, helm6 as H
    build.build()
    prob = O.Problem(n, 0.3 * (n + 1) * (1 + 0.02j), faces)
    x = inputs.complex_normal(n, prob.shape)
    ref = O.Preconditioner(prob)(x)
    for _ in range(3):
        fill = [torch.full((1 << m,), float("nan"), device="cuda") for m in (16, 18, 20, 22, 24, 26)]
        torch.cuda.synchronize()
        del fill
        torch.cuda.empty_cache()  # back to the driver, which gives it to the next context
        with H.Solver(n, prob.k, faces, precision=H.MIXED, method=H.FGMRES) as s:
            y = s.apply_Pinv(torch.from_numpy(x).cuda()).cpu().numpy()
        # the mixed preconditioner's tolerance (BF16-split transforms, FP32 accumulation)
        assert np.abs(y - ref).max() <= 1e-4 * np.abs(ref).max()
