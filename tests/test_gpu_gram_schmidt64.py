"""The FP64 Gram-Schmidt update pass by itself (launch_dcgs_update<double, double>),
    v = (u - sum_i V_i s_i) / alpha,   u' = (w - sum_i V_i t_i - v c) / alpha,
against extended precision.  The sum over V_i s_i has two forms: FP64, and FP32 where every |s_i| is below
2^-36 alpha.  Cases on both sides of that line, one large coefficient among small ones, basis values that
vanish in FP32, alpha far from 1 (where FP32's exponents would not reach), one and two points per thread, up
to 64 vectors (more than the kernel holds at once)."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U = 2.0 ** -53


def update(lib, V, u, w, s, t, c, alpha):
    count, N = V.shape
    f = getattr(lib, "_ZN5helm618launch_dcgs_updateIddEEvPKT0_liPT_PKS4_PS1_lPKdidP11CUstream_st")
    P = C.c_void_p
    f.argtypes, f.restype = [P, C.c_int64, C.c_int, P, P, P, C.c_int64, P, C.c_int, C.c_double, P], None
    planar = lambda a: torch.from_numpy(np.concatenate([a.real, a.imag])).cuda()
    dV = torch.from_numpy(np.concatenate([V.real, V.imag], axis=1)).cuda()
    du, dw, dv = planar(u), planar(w), torch.zeros(2 * N, dtype=torch.float64, device="cuda")
    pairs = lambda a: np.stack([a.real, a.imag], axis=1).ravel()
    coef = torch.from_numpy(np.concatenate([pairs(s), pairs(t), [c.real, c.imag, 1.0 / alpha]])).cuda()
    f(dV.data_ptr(), 2 * N, count, du.data_ptr(), dw.data_ptr(), dv.data_ptr(), N, coef.data_ptr(), 24, 1.0,
      torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    h = lambda a: a[:N].cpu().numpy() + 1j * a[N:].cpu().numpy()
    return h(dv), h(du)


def data(N, count, size, alpha):
    """size: |s_i| / alpha, or "one" (a single coefficient of 0.3 alpha)."""
    g = np.random.default_rng(N + count)
    z = lambda *sh: g.standard_normal(sh) + 1j * g.standard_normal(sh)
    V = z(count, N) / np.sqrt(2.0 * N)
    V[:, 3] = 0.0
    V[:, 4] *= 2.0 ** -140  # below FP32's normal numbers
    V[:, 5] *= 2.0 ** -1040
    u, w = alpha * z(N) / np.sqrt(2.0 * N), z(N)
    s = z(count)
    s *= alpha * (2.0 ** -40 if size == "one" else size) / np.abs(s).max()
    if size == "one":
        s[count // 2] = alpha * (0.3 - 0.1j)
    return V, u, w, s, 0.1 * z(count), 0.7 - 0.2j


@pytest.mark.parametrize("alpha", [0.37, 2.0 ** -200, 2.0 ** 200])
@pytest.mark.parametrize("size", [0.0, 2.0 ** -52, 0.9 * 2.0 ** -37, 1.1 * 2.0 ** -36, 2.0 ** -20, 0.5, "one"])
@pytest.mark.parametrize("N,count", [(4096, 1), (1001, 30), (4098, 33), (1001, 64), (4098, 64)])
def test_update_pass(N, count, size, alpha):
    from paper_1212_1397_gb300 import build, helm6
    build.build()
    V, u, w, s, t, c = data(N, count, size, alpha)
    v, un = update(helm6.load(), V, u, w, s, t, c, alpha)
    L = np.clongdouble
    inv = np.longdouble(1.0 / alpha)  # what the kernel is given
    rv = (u.astype(L) - s.astype(L) @ V.astype(L)) * inv
    ru = (w.astype(L) - t.astype(L) @ V.astype(L) - v.astype(L) * L(c)) * inv
    # v: 2 count + 2 roundings, each of a partial sum no larger than |u| + sum |V_i| |s_i|
    part = np.abs(u) + np.abs(s) @ np.abs(V)
    ev = np.abs(v - rv) * alpha
    assert np.all(ev <= (2 * count + 3) * U * part + 1e-320)
    if alpha == 0.37 and size != "one" and size < 2.0 ** -36:
        # the FP32 form: in each component one rounding of the difference and one of the scaling; the sum in FP32 (values cut
        # to 24 bits, 2 count roundings of a partial sum)
        assert np.all(ev <= 3 * U * np.abs(u) + (2 * count + 4) * 2.0 ** -23 * (np.abs(s) @ np.abs(V)) + 1e-320)
    part = np.abs(w) + np.abs(t) @ np.abs(V) + np.abs(v) * abs(c)
    assert np.all(np.abs(un - ru) * alpha <= (2 * count + 6) * U * part)
