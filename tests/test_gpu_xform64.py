"""FP64 transforms in integer slices on the tensor cores (what an FP64 context with the form left
to the library uses from 8,192 unknowns on): A_p^-1 against the oracle and against the FFT-type
and dense forms, over face pairs (folded and unfolded bases), axis lengths around the stages of
16 points, the groups of 128 modes, the tiles of 128 rows and the odd lengths that copy 8 bytes
at a time; rows whose values span the exponent range; zero, denormal and non-finite rows."""
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


def pinv(H, n, k, faces, x, transform="auto"):
    with H.Solver(n, k, faces, precision=H.FP64, method=H.SKS, transform=transform) as s:
        return s.apply_Pinv(torch.from_numpy(x).cuda()).cpu().numpy()


@pytest.mark.parametrize("n,faces", [(20, "DDNNSS"), (21, "NNDDDS"), (31, "DNNDSS"), (32, "NDDNNN"),
                                     (33, "DDNDSD"), (47, "NNNNSS"), (64, "NDNNDD")])
def test_matches_oracle(H, n, faces):
    k = 0.2 * (n + 1) * (1 + 0.3j)  # damped: the z lines amplify a transform's rounding by a few units
    prob = O.Problem(n, k, faces)
    x = inputs.complex_normal(n, prob.shape)
    ref = O.Preconditioner(prob)(x)
    # a few roundings of 2^-53 per transform and line, LAPACK's own included: 1e-12 of the maximum
    assert np.abs(pinv(H, n, k, faces, x) - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("n,faces", [(126, "DDNNSS"), (127, "DDDDDD"), (128, "NNDDSS"), (129, "DDNNSD"),
                                     (130, "NDDNSS"), (191, "DDNDSS")])
def test_matches_other_forms(H, n, faces):
    k = 0.2 * (n + 1) * (1 + 0.3j)
    x = inputs.complex_normal(n, O.Problem(n, k, faces).shape)
    ref = pinv(H, n, k, faces, x, "fft")  # FFT-type where the length has one, else dense
    # the dense form's basis entries carry an argument rounding of up to m^2 2^-53 pi: 1e-11
    assert np.abs(pinv(H, n, k, faces, x) - ref).max() <= 1e-11 * np.abs(ref).max()


@pytest.mark.parametrize("scale", [1e-300, 1e-150, 1e150])
def test_scales(H, scale):
    """A power of ten in front of the field is one behind the result (the rows' own scales)."""
    n, k, faces = 31, 6 + 2j, "DDNNSS"
    x = inputs.complex_normal(3, O.Problem(n, k, faces).shape)
    a, b = pinv(H, n, k, faces, x), pinv(H, n, k, faces, scale * x)
    # 1e-300 leaves about 2^-52 of a row above the smallest normal number's last bit
    assert np.abs(b / scale - a).max() <= 1e-13 * np.abs(a).max()


def test_rows_of_mixed_size(H):
    """Neighbouring rows 200 decades apart, zero planes and a constant row at the top of a binade (the
    sum of two points then needs the digits' last bit)."""
    n, k, faces = 31, 6 + 2j, "DDNNSS"
    prob = O.Problem(n, k, faces)
    x = inputs.complex_normal(4, prob.shape)
    x[5] = 0.0
    x[7, 3] *= 1e-200
    x[9, 4] = 2.0 - 2.0 ** -52
    x[11].imag = 0.0
    ref = O.Preconditioner(prob)(x)
    assert np.abs(pinv(H, n, k, faces, x) - ref).max() <= 1e-12 * np.abs(ref).max()
    assert not np.any(pinv(H, n, k, faces, np.zeros_like(x)))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_rows_stay_non_finite(H, bad):
    n, k, faces = 31, 6 + 2j, "DDNNSS"
    x = inputs.complex_normal(5, O.Problem(n, k, faces).shape)
    x[4, 5, 6] = bad
    assert not np.isfinite(pinv(H, n, k, faces, x)).all()


@pytest.mark.parametrize("n,faces", [(127, "DNNDSS"), (128, "DNNDDD"), (129, "NDNDSS"), (131, "NDNDSS"), (255, "NNDDSS"), (256, "DDNNSS"),
                                     (258, "NNNNSD"), (259, "NNDDSS")])
def test_modes_beyond_whole_groups(H, n, faces):
    """Axes one to five modes longer than whole groups of 128 (128, 130 and 132 modes of a quarter-wave axis, 257,
    258, 260 and 261 of a cosine one): up to two are formed apart in FP64."""
    k = 0.2 * (n + 1) * (1 + 0.3j)
    prob = O.Problem(n, k, faces)
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.view_as_complex(torch.randn(prob.shape + (2,), dtype=torch.float64, device="cuda", generator=gen))
    out = []
    for form in ("auto", "fft"):
        with H.Solver(n, k, faces, precision=H.FP64, method=H.SKS, transform=form) as s:
            out.append(s.apply_Pinv(x))
    # as above: the dense form's basis entries carry an argument rounding
    assert float((out[0] - out[1]).abs().max()) <= 1e-11 * float(out[1].abs().max())


@pytest.mark.parametrize("eps", [0.0, 1e-18, 1e-9, 1e-4])
def test_smooth_rows(H, eps):
    """Rows of one low mode (and eps of noise): nearly all results are integers far below a row's scale,
    down to single units and zeros; to a few roundings of the largest, like any other row."""
    n, k, faces = 63, 12 + 4j, "DDNNSS"
    prob = O.Problem(n, k, faces)
    mz, my, mx = prob.shape
    x = (np.sin(np.pi * np.arange(1, mx + 1) / (n + 1))[None, None, :] * np.cos(np.pi * np.arange(my) / (n + 1))[None, :, None]
         * np.exp(-np.arange(mz) / 9.0)[:, None, None]).astype(np.complex128) * (1 - 0.5j)
    x = x + eps * inputs.complex_normal(7, prob.shape)
    ref = O.Preconditioner(prob)(x)
    assert np.abs(pinv(H, n, k, faces, x) - ref).max() <= 1e-12 * np.abs(ref).max()
