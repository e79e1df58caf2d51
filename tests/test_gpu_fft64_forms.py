"""The FP64 FFT-type transforms against the oracle, asked for by name (with the form left to the library a
context of 8,192 unknowns or more takes the integer-slice form): the lengths and face pairs of
test_gpu_fft, and the dense form where there is no FFT."""
import numpy as np
import pytest

import helm6_inputs as inputs
import oracle as O

from test_gpu_fft import FFT_CASES, H, relmax  # noqa: F401 (H is a fixture)

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,faces,form", [c + ("fft",) for c in FFT_CASES]
                         + [(24, "DDNNSS", "dense"), (63, "DNNDSS", "dense"), (100, "DDNNSS", "dense")])
def test_named_form_matches_oracle(H, n, faces, form):  # noqa: F811
    k = 9.0 + 0.3j
    prob = O.Problem(n, k, faces)
    x = inputs.complex_normal(700 + n, prob.shape)
    with H.Solver(n, k, faces, precision=H.FP64, transform=form) as s:
        assert s.transforms == (form, form)
        y = s.apply_Pinv(torch.from_numpy(x).cuda()).cpu().numpy()
    # as for the other forms: the z lines amplify rounding by the line's condition number
    assert relmax(y, O.Preconditioner(prob)(x)) < 1e-10
