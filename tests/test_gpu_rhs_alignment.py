"""The right side's arrays: a caller's F and noise may begin on any double (the C interface takes
plain device pointers), not only on 16 bytes; the result is the same as for aligned arrays."""
import ctypes as C

import numpy as np
import pytest

import helm6_inputs as inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def H():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1212_1397_gb300 import build, helm6
    build.build()
    return helm6


@pytest.mark.parametrize("off_F,off_noise", [(0, 1), (1, 0), (1, 1), (1, None)])
@pytest.mark.parametrize("n,nsrc", [(5, 1), (33, 40)])  # 40 terms: a second pass reads F again
def test_arrays_on_any_double(H, n, nsrc, off_F, off_noise):
    src = inputs.gaussian_sources(5, n, nsrc, margin_h=1)
    with H.Solver(n, 4.0 + 0.2j, "DNNDSS", method=H.SKS) as s:
        N = int(np.prod(s.shape))
        noise = torch.from_numpy(inputs.complex_normal(9, s.shape)).cuda()
        ref = s.rhs_gaussians(src, noise=None if off_noise is None else noise)
        F = torch.zeros(2 * N + 1, dtype=torch.float64, device="cuda")
        nz = torch.zeros(2 * N + 1, dtype=torch.float64, device="cuda")
        ptr = None
        if off_noise is not None:
            nz[off_noise:off_noise + 2 * N] = torch.view_as_real(noise).reshape(-1)
            ptr = C.c_void_p(nz.data_ptr() + 8 * off_noise)
        assert F.data_ptr() % 16 == 0 and nz.data_ptr() % 16 == 0
        cen = (C.c_double * (3 * nsrc))(*src.centers.ravel().tolist())
        amps = (H.C64 * nsrc)(*[H.C64(a.real, a.imag) for a in src.amps])
        rc = H.load().helm6_rhs_gaussians(s._ctx, nsrc, cen, amps, float(src.sigma), ptr, C.c_void_p(F.data_ptr() + 8 * off_F))
        torch.cuda.synchronize()
    assert rc == 0
    assert torch.equal(F[off_F:off_F + 2 * N], torch.view_as_real(ref).reshape(-1))
    assert float(F[2 * N * (1 - off_F)]) == 0.0  # the double beside the array is untouched
