"""The FP64 operator at the edges of its 16 x 32 tiles and z chunks, against the oracle.

Sizes with one point more or less than a tile, a warp's four rows or a thread's two points per axis;
one chunk and many; every kind of face; real and complex wavenumbers (their kernels differ); the
caller's arrays apart (read and written in place), overlapping (through planar copies) and with
Sommerfeld-like faces off z (axes exchanged); the residual with its norm.

A result sums 27 products in chains of at most about 20 roundings of 2^-53; with |u| around 1 the
terms' magnitudes add up to less than 40 where the largest result is above 5: 1e-13 of it.
"""
import numpy as np
import pytest

import helm6_inputs as inputs
import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [(3, 2.0, "DDDDDD"), (5, 3.0 + 0.4j, "NNNNNN"), (14, 4.0, "DNNDSS"), (15, 5.0 + 0.3j, "DDNNSD"),
         (16, 5.0, "NNDDDS"), (17, 6.0 + 0.2j, "DDDDSS"), (30, 9.0, "DDNNSS"), (31, 9.0 + 0.2j, "NDDNNN"),
         (33, 9.0, "NDDNND"), (47, 8.0 + 0.1j, "DDDDDN"), (66, 12.0, "DDNNSS")]


def _close(a, b):
    return np.abs(a - b).max() <= 1e-13 * np.abs(b).max()


@pytest.mark.parametrize("n,k,faces", CASES)
def test_operator_and_residual(n, k, faces):
    from paper_1212_1397_gb300 import build, helm6 as H
    build.build()
    prob = O.Problem(n, k, faces)
    u = inputs.complex_normal(51, prob.shape)
    F = inputs.complex_normal(52, prob.shape)
    ref = O.apply_A(prob, u)
    ud, Fd = torch.from_numpy(u).cuda(), torch.from_numpy(F).cuda()
    with H.Solver(n, k, faces, precision=H.FP64) as s:
        assert _close(s.apply_A(ud).cpu().numpy(), ref)
        buf = torch.zeros(2 * u.size, dtype=torch.complex128, device="cuda")  # y one point behind x
        x, y = buf[1:1 + u.size].view(prob.shape), buf[:u.size].view(prob.shape)
        x.copy_(ud)
        assert _close(s.apply_A(x, y).cpu().numpy(), ref)
        x.copy_(ud)
        assert _close(s.apply_A(x, x).cpu().numpy(), ref)
    r, ss = torch.empty_like(ud), torch.empty(1, dtype=torch.float64, device="cuda")
    assert H.residual_noalloc(n, k, faces, Fd, ud, r, ss) == 0
    rn = F - ref
    assert _close(r.cpu().numpy(), rn)
    assert abs(float(ss[0]) - float((np.abs(rn) ** 2).sum())) <= 1e-12 * float((np.abs(rn) ** 2).sum())


def test_operator_with_radiating_x_faces():
    from paper_1212_1397_gb300 import helm6 as H
    n, k = 21, 6.0 + 0.2j
    u = torch.from_numpy(inputs.complex_normal(53, (n, n, n + 2))).cuda()  # Sommerfeld-like faces on x
    with H.Solver(n, k, "SSDDDD", precision=H.FP64) as s, H.Solver(n, k, "DDDDSS", precision=H.FP64) as t:
        a = s.apply_A(u).cpu().numpy()
        b = t.apply_A(u.permute(2, 1, 0).contiguous()).permute(2, 1, 0).cpu().numpy()
    assert _close(a, b)
