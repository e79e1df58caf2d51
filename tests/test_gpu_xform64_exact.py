"""One FP64 integer-slice transform by itself (launch_xform64) against extended precision: every digit level's
path out of the accumulators, sums above 2^22 among them, for folded and unfolded axes up to the largest the
form takes, both stores and a last tile that is not full; and what a context does where an axis is out of
the form's range."""
import ctypes as C
import math

import numpy as np
import pytest

import helm6_inputs as inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


class Basis(C.Structure):  # helm6::X64Basis
    _fields_ = [("dev", C.c_void_p), ("bytes", C.c_size_t), ("planes", C.c_size_t)] + [
        (f, C.c_int) for f in ("m", "fold", "nk", "nch", "gcols", "ngroups", "eb", "tail")]


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1212_1397_gb300 import build, helm6
    build.build()
    return helm6.load()


def matrix(n, lo, hi, inverse):
    """(trigonometric table, transform matrix) of an axis, in doubles."""
    nlo, nhi = lo != "D", hi != "D"
    N, m = n + 1, n + nlo + nhi
    D = 2 * N if nlo != nhi else N
    fn = math.cos if nlo else math.sin
    trig = np.array([fn(math.pi * q / D) for q in range(2 * D)])
    if nlo:
        trig[[D // 2, 3 * D // 2]] *= D % 2  # exact zeros
    else:
        trig[[0, D]] = 0.0
    node = np.arange(m) + (0 if nlo else 1)
    mode = 2 * np.arange(m) + 1 if nlo != nhi else np.arange(m) + (0 if nlo else 1)
    V = trig[np.outer(node, mode) % (2 * D)]
    if inverse:
        return trig, V
    w, wm = np.ones(m), np.ones(m)
    w[(node == 0) & nlo] = 0.5
    w[(node == N) & nhi] = 0.5
    if nlo and nhi:
        wm[(mode == 0) | (mode == N)] = 0.5
    return trig, (2.0 / N) * (wm[:, None] * w[None, :]) * V.T


def digits(b, eb):
    """The seven balanced base-256 digits of an array on the scale 2^(eb - 55)."""
    x = np.rint(np.ldexp(b, 55 - eb)).astype(np.int64)
    out = []
    for d in range(6, -1, -1):
        v = ((x + 128) & 255) - 128 if d else x
        x = (x - v) >> 8
        out.insert(0, v)
    return out


def transform(lib, n, lo, hi, inverse, x, transposed=0, R=1):
    trig, B = matrix(n, lo, hi, inverse)
    code = {"D": 0, "N": 1}
    plan = getattr(lib, "_ZN5helm68x64_planEiii")
    plan.argtypes, plan.restype = [C.c_int] * 3, Basis
    h = plan(n, code[lo], code[hi])
    conf = getattr(lib, "_ZN5helm613x64_configureEv")
    conf.restype = C.c_int
    assert conf() == 0 and h.m == B.shape[0]
    store = torch.zeros(h.bytes, dtype=torch.uint8, device="cuda")
    h.dev = store.data_ptr()
    flags = torch.zeros(2, dtype=torch.int32, device="cuda")
    dt = torch.from_numpy(trig).cuda()
    st = torch.cuda.current_stream().cuda_stream
    fill = getattr(lib, "_ZN5helm617launch_x64_digitsEiiiiRNS_8X64BasisEPKdPiP11CUstream_st")
    fill.argtypes, fill.restype = [C.c_int] * 4 + [C.POINTER(Basis)] + [C.c_void_p] * 3, None
    fill(n, code[lo], code[hi], inverse, C.byref(h), dt.data_ptr(), flags.data_ptr(), st)
    go = getattr(lib, "_ZN5helm614launch_xform64ERKNS_8X64BasisEPKdPdiiiPiP11CUstream_stii")
    go.argtypes = [C.POINTER(Basis), C.c_void_p, C.c_void_p] + [C.c_int] * 3 + [C.c_void_p, C.c_void_p, C.c_int, C.c_int]
    go.restype = None
    rows, m = x.shape
    ld = m + (m & 1)
    src = torch.full((rows, ld), float("nan"), dtype=torch.float64, device="cuda")  # the padding is not read
    src[:, :m] = torch.from_numpy(x).cuda()
    if transposed:
        out = torch.zeros((rows // R, m, R), dtype=torch.float64, device="cuda")
        go(C.byref(h), src.data_ptr(), out.data_ptr(), rows, 1, R, flags[1:].data_ptr(), st, ld, R)
    else:
        out = torch.zeros((rows, ld), dtype=torch.float64, device="cuda")
        go(C.byref(h), src.data_ptr(), out.data_ptr(), rows, 0, 1, flags[1:].data_ptr(), st, ld, ld)
    torch.cuda.synchronize()
    assert flags.tolist() == [0, 0]  # the axis is in range, no wait ran out
    y = out.cpu().numpy()
    return h, B, (y.transpose(0, 2, 1).reshape(rows, m) if transposed else y[:, :m])


def check(h, B, x, y):
    ref = x.astype(np.longdouble) @ B.T.astype(np.longdouble)
    # per point, in units of the row's largest value and of the basis' bound 2^eb: the data cut to 2^-52 and the
    # basis rounded to 2^-56, the digit pairs left out (six of 2^14 at level 7 on the scale 2^-109 2^56: 2^-52.4, each
    # further level 2^-8 of that); and one rounding of the result
    big = np.abs(x).max(axis=1, keepdims=True)
    bound = x.shape[1] * 2.0 ** -51 * big * 2.0 ** h.eb + 2.0 ** -52 * np.abs(ref)
    assert np.all(np.abs(y - ref) <= bound)


# unfolded up to the limit (a quarter-wave axis of 255 points is in range, 263 is not), folded to several groups
AXES = [(20, "D", "D"), (31, "D", "N"), (63, "N", "N"), (129, "N", "D"), (248, "D", "N"), (300, "D", "D"),
        (330, "N", "N"), (400, "D", "D"), (460, "N", "N"), (540, "D", "D")]


@pytest.mark.parametrize("inverse", [0, 1])
@pytest.mark.parametrize("n,lo,hi", AXES)
def test_rows_of_all_kinds(lib, n, lo, hi, inverse):
    """Random rows, rows that fall off over thirty decades, single points, a constant and zero."""
    m = n + (lo != "D") + (hi != "D")
    g = np.random.default_rng(n)
    x = g.standard_normal((130, m))
    x[1::5] *= 10.0 ** -np.linspace(0.0, 30.0, m)
    x[2] = 0.0
    x[3] = 0.0
    x[3, m // 3] = -1.75
    x[4] = 1.0
    x[5] *= 1e-200
    h, B, y = transform(lib, n, lo, hi, inverse, x)
    check(h, B, x, y)
    h, B, yt = transform(lib, n, lo, hi, inverse, x, transposed=1, R=10)
    assert np.array_equal(y, yt)


@pytest.mark.parametrize("inverse", [0, 1])
@pytest.mark.parametrize("n,lo,hi", [(248, "D", "N"), (248, "N", "D"), (400, "D", "D"), (460, "N", "N"), (540, "D", "D")])
def test_level_sums_above_2_22(lib, n, lo, hi, inverse):
    """Rows whose digits follow the signs of a mode's digits, so that its level-2 sum comes near the largest
    there can be (above 2^22 it leaves the accumulator through the general conversion)."""
    _, B = matrix(n, lo, hi, inverse)
    m, fold = B.shape[0], lo == hi
    eb = 0
    while not inverse and math.ldexp(1.0, eb - 1) >= 2.0 / (n + 1):
        eb -= 1
    g = np.random.default_rng(n)
    x = g.standard_normal((140, m))
    x /= np.abs(x).max(axis=1, keepdims=True)
    reached = 0
    for r in range(0, 128, 2):
        p = int(g.integers(0, m))
        half = B[p, : (m + 1) // 2] if fold else B[p]
        b = digits(half, eb)
        if fold and m % 2:
            for d in b:
                d[-1] = 0
        sg = [np.where(b[2 - i] < 0, -1, 1) for i in range(3)]
        a0 = 126 if fold else 62  # digits of the sum of a point and its mirror image, or of a point
        v = a0 * sg[0] * 2 ** 48 + 127 * sg[1] * 2 ** 40 + 127 * sg[2] * 2 ** 32
        s2 = int((a0 * sg[0] * b[2] + 127 * sg[1] * b[1] + 127 * sg[2] * b[0]).sum())
        reached = max(reached, abs(s2))
        f = np.ldexp(v.astype(np.float64), -55 if fold else -54)
        if fold:
            x[r, : len(f)] = f
            x[r, m - len(f):][::-1] = f * (1 if p % 2 == 0 else -1)
            if m % 2:
                x[r, m // 2] = 0.0
        else:
            x[r] = f
    assert reached > 2 ** 22  # the case is one
    h, B, y = transform(lib, n, lo, hi, inverse, x)
    assert h.eb == eb
    check(h, B, x, y)


@pytest.mark.parametrize("n,faces", [(255, "DNDDSS"), (263, "DNDDSS"), (264, "DDNDSS"), (300, "DDNNSS"), (320, "DDDNSS")])
def test_contexts_around_the_range(n, faces, lib):
    """A_p^-1 where an axis is near the form's range or beyond it (a quarter-wave axis of 263 or 320 points:
    the whole context takes the other forms) against the other forms, and no memory kept for what is not used."""
    from paper_1212_1397_gb300 import helm6 as H
    k = 0.2 * (n + 1) * (1 + 0.3j)
    out, used = [], []
    for form in ("fft", "auto", "fft", "auto"):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        with H.Solver(n, k, faces, precision=H.FP64, method=H.SKS, transform=form) as s:
            used.append(before - torch.cuda.mem_get_info()[0])
            gen = torch.Generator(device="cuda").manual_seed(n)
            x = torch.view_as_complex(torch.randn(s.shape + (2,), dtype=torch.float64, device="cuda", generator=gen))
            out.append(s.apply_Pinv(x))
    # the dense form's basis entries carry an argument rounding of up to m^2 2^-53 pi: 1e-11
    assert float((out[1] - out[0]).abs().max()) <= 1e-11 * float(out[0].abs().max())
    if n in (263, 320):
        assert torch.equal(out[3], out[2])  # the same kernels
        assert used[3] <= used[2] + (2 << 20), used  # the driver hands out memory in pieces of 2 MiB
