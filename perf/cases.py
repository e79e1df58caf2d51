"""What a user of the solver has it do, as cases that can be timed.

A case is a dict of plain values; `kind` says which entry point it calls:

    solve     Solver.solve: one complete solve from u = 0 (the whole call, host loop included)
    batch     solve_batch: several independent problems of uneven size
    pinv      Solver.apply_Pinv: the 7-point preconditioner's direct inverse
    apply     Solver.apply_A: the sixth-order operator
    residual  residual_noalloc: F - A u and its norm without a context
    rhs       Solver.rhs_gaussians: the compact right side
    gradient  Trainer.gradient: loss and parameter gradient of the learned stage's network

Sizes, faces, wavenumbers and options are those of the workloads (helm6_inputs.WORKLOADS,
batch_problems), of the paper's tables and of the tests.  Solves in mixed precision ask for the
accuracy of an FP64 solve (1e-12), so that u is determined to well below a solve's own rounding.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import helm6_inputs as inputs
from paper_1212_1397_gb300 import helm6 as H

RESTART = 30


def listed():
    return [
        # the bench workload: the largest mixed solve, one device-driven graph
        dict(name="solve_mixed_n256", kind="solve", n=256, kr=80.0, ki=0.0, faces="DDNNSS", precision="mixed",
             method="fgmres", restart=30, graphs=2, tol=1e-12, nsrc=8, noise=0.0),
        # the mid-size mixed workload, options left at their defaults (host-driven), GMRES(20)
        dict(name="solve_mixed_n128", kind="solve", n=128, kr=40.0, ki=0.0, faces="DDNNSS", precision="mixed",
             method="fgmres", restart=20, graphs=0, tol=1e-12, nsrc=1, noise=1e-3),
        # the smallest solves a program makes: launches and hand-overs between kernels count
        dict(name="solve_mixed_n32", kind="solve", n=32, kr=10.0, ki=0.1, faces="DDDDDD", precision="mixed",
             method="fgmres", restart=20, graphs=2, tol=1e-12, nsrc=1, noise=0.0),
        # several problems of uneven size and faces in one call
        dict(name="batch_6", kind="batch", count=6, seed=0, tol=1e-12),
        # the library's default solver (FP64 GMRES) on the paper's Dirichlet cube, h = 1/128
        dict(name="solve_fp64_n127", kind="solve", n=127, kr=30.0, ki=0.0, faces="DDDDDD", precision="fp64",
             method="gmres", restart=30, graphs=0, tol=1e-10, nsrc=1, noise=0.0),
        # Algorithm 1 at the paper's finest tabulated grid of Table 4, h = 1/256
        dict(name="sks_fp64_n255", kind="solve", n=255, kr=30.0, ki=0.0, faces="DDDDDD", precision="fp64",
             method="sks", restart=30, graphs=0, tol=1e-10, nsrc=1, noise=0.0),
        # FP64 GMRES on a grid whose axes have no FFT-type transform (n + 1 = 193), mixed quarter-wave faces
        dict(name="solve_fp64_n192", kind="solve", n=192, kr=20.0, ki=0.2, faces="DNNDSS", precision="fp64",
             method="gmres", restart=30, graphs=0, tol=1e-10, nsrc=1, noise=1e-3),
        # the preconditioner and the operator alone, for a user's own Krylov method
        dict(name="pinv_fp64_n256", kind="pinv", n=256, kr=80.0, ki=0.0, faces="DDNNSS"),
        dict(name="apply_fp64_n100", kind="apply", n=100, kr=30.0, ki=0.3, faces="DNNNSS"),
        # residual check inside a runtime that owns the device memory
        dict(name="residual_n256", kind="residual", n=256, kr=80.0, ki=0.0, faces="DDNNSS"),
        # setting up a problem: the compact right side of eight sources and a noise field
        dict(name="rhs_n256", kind="rhs", n=256, kr=80.0, ki=0.0, faces="DDNNSS", nsrc=8, noise=1e-3),
        # one training step's gradient of the learned stage, batch of 32^3 patches
        dict(name="gradient_b32", kind="gradient", batch=32, side=32, kh=0.31),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the whole range of each kind, odd and ragged ones among them."""
    kind = rng.choice(["solve", "solve", "solve", "batch", "pinv", "pinv", "apply", "residual", "rhs", "gradient"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 5), seed=rng.randint(1, 10 ** 6), tol=1e-12)
    if kind == "gradient":
        return dict(kind=kind, batch=rng.randint(2, 32), side=rng.choice([16, 24, 31, 32]), kh=0.31)
    xy = "".join(rng.choice("DN") for _ in range(4))
    z = rng.choice(["SS", "SS", "DS", "SN", "DD", "NN", "DN"])
    n = _log_int(rng, 24, 250)
    # the resolution range of the workloads (kh up to 0.31); absorption where no face radiates
    kr = rng.uniform(0.05, 0.31 if kind != "solve" else 0.2) * (n + 1)
    ki = 0.01 * kr if ("S" not in z or rng.random() < 0.5) else 0.0
    base = dict(kind=kind, n=n, kr=kr, ki=ki, faces=xy + z)
    if kind == "solve":
        mixed = rng.random() < 0.6
        base.update(precision="mixed" if mixed else "fp64", method="fgmres" if mixed else "gmres",
                    restart=rng.choice([20, 30]), graphs=rng.choice([0, 2]) if mixed else 0,
                    tol=1e-12 if mixed else 1e-10, nsrc=rng.randint(1, 8), noise=rng.choice([0.0, 1e-3]))
    if kind == "rhs":
        base.update(nsrc=rng.randint(1, 16), noise=rng.choice([0.0, 1e-3]))
    return base


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------

def _problems(case):
    """Problem descriptions of a batch, sizes drawn over the batched workload's own."""
    return inputs.batch_problems(case["seed"], case["count"])


def _field(shape, seed, scale=1.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.empty(tuple(shape) + (2,), dtype=torch.float64, device="cuda").normal_(generator=g)
    return torch.view_as_complex(x.mul_(scale / math.sqrt(2.0)))


def _solver(case):
    mixed = case.get("precision", "fp64") == "mixed"
    method = {"gmres": H.GMRES, "fgmres": H.FGMRES, "sks": H.SKS}[case.get("method", "sks")]
    return H.Solver(case["n"], complex(case["kr"], case["ki"]), case["faces"], precision=H.MIXED if mixed else H.FP64,
                    method=method, max_restart=case.get("restart", RESTART), use_graphs=case.get("graphs", 0))


def _sources(case, seed):
    return inputs.gaussian_sources(seed, case["n"], case["nsrc"], margin_h=min(16, max(1, case["n"] // 4)))


def _noise(case, seed, shape):
    return _field(shape, seed + 1, case["noise"]) if case["noise"] else None


def _batch_sources(p, seed):
    return inputs.gaussian_sources(p["src_seed"] + 7919 * seed, p["n"], 1, margin_h=4)


def _dims(n, faces):
    return inputs.dims(n, faces)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        # a batch's contexts with the grids of the default schedule, right sides in place
        items = []
        for p in _problems(case):
            s = H.Solver(p["n"], p["k"], p["faces"], precision=H.MIXED, method=H.FGMRES, max_restart=RESTART,
                         own_stream=True, use_graphs=2)
            items.append((s, s.rhs_gaussians(_batch_sources(p, seed))))
        torch.cuda.synchronize()
        return dict(kind=kind, solvers=[i[0] for i in items], F=[i[1] for i in items], tol=case["tol"],
                    u=[s.empty() for s, _ in items])
    if kind == "gradient":
        b, m = case["batch"], case["side"]
        g = np.random.default_rng(seed)
        theta = []
        for ci, co in zip((2, 16, 16, 16), (16, 16, 16, 2)):
            theta += [g.standard_normal(co * ci * 27) * math.sqrt(2.0 / (27 * ci)), 0.05 * g.standard_normal(co)]
        theta = np.concatenate(theta).astype(np.float32)
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        x = torch.empty((b, m, m, m, 2), dtype=torch.float32, device="cuda").normal_(generator=gen)
        t = H.Trainer(b, m, m, m, theta)
        t.set_residual_loss(case["kh"] * 129, 1.0 / 129)
        return dict(kind=kind, trainer=t, x=x)
    if kind == "residual":
        mx, my, mz = _dims(case["n"], case["faces"])
        F, u = _field((mz, my, mx), seed), _field((mz, my, mx), seed + 1)
        return dict(kind=kind, n=case["n"], k=complex(case["kr"], case["ki"]), faces=case["faces"], F=F, u=u,
                    r=torch.empty_like(F), ss=torch.zeros(1, dtype=torch.float64, device="cuda"))
    s = _solver(case)
    if kind in ("pinv", "apply"):
        x = _field(s.shape, seed)
        return dict(kind=kind, s=s, x=x, y=torch.empty_like(x))
    src = _sources(case, seed)
    noise = _noise(case, seed, s.shape)
    if kind == "rhs":
        return dict(kind=kind, s=s, src=src, noise=noise, F=s.empty())
    return dict(kind=kind, s=s, F=s.rhs_gaussians(src, noise=noise), u=s.empty(), tol=case["tol"],
                restart=case["restart"])


def run(state):
    kind = state["kind"]
    if kind == "solve":
        u = state["u"].zero_()
        _, st = state["s"].solve(state["F"], u=u, tol=state["tol"], restart=state["restart"], maxit=2000)
        return dict(u=u, rc=int(st["rc"]))
    if kind == "batch":
        for u in state["u"]:
            u.zero_()
        rc, _ = H.solve_batch(state["solvers"], state["F"], state["u"], tol=state["tol"], restart=RESTART, maxit=2000)
        return dict(u=state["u"], rc=int(rc))
    if kind == "pinv":
        return state["s"].apply_Pinv(state["x"], state["y"])
    if kind == "apply":
        return state["s"].apply_A(state["x"], state["y"])
    if kind == "residual":
        H.residual_noalloc(state["n"], state["k"], state["faces"], state["F"], state["u"], state["r"], state["ss"])
        return dict(r=state["r"], sumsq=state["ss"])
    if kind == "rhs":
        return state["s"].rhs_gaussians(state["src"], noise=state["noise"], F=state["F"])
    loss, grad = state["trainer"].gradient(state["x"], state["x"])
    return dict(loss=float(loss), grad=grad)


def work(case):
    """Every input read once and every output written once; the arithmetic of one application of
    what the call cannot do without (a solve: at least one operator and one preconditioner)."""
    kind = case["kind"]
    if kind == "gradient":
        pts = case["batch"] * case["side"] ** 3
        taps = 27 * (2 * 16 + 16 * 16 + 16 * 16 + 16 * 2)
        return dict(bytes=8.0 * pts + 8.0 * H.CNN_NPARAMS, flops=6.0 * taps * pts)
    if kind == "batch":
        ws = [work(dict(kind="solve", n=p["n"], faces=p["faces"])) for p in _problems(case)]
        return dict(bytes=sum(w["bytes"] for w in ws), flops=sum(w["flops"] for w in ws))
    N = float(np.prod(_dims(case["n"], case["faces"])))
    lg = math.log2(case["n"] + 2)
    pinv, op = N * (4 * 5 * lg + 28), N * 60
    if kind == "pinv":
        return dict(bytes=32.0 * N, flops=pinv)
    if kind == "apply":
        return dict(bytes=32.0 * N, flops=op)
    if kind == "residual":
        return dict(bytes=48.0 * N, flops=op + 6 * N)
    if kind == "rhs":
        return dict(bytes=16.0 * N * (2 if case["noise"] else 1), flops=12.0 * N * case["nsrc"])
    return dict(bytes=32.0 * N, flops=pinv + op)


# ---------------------------------------------------------------------------------------
# the same results in 64 bits from plain torch
# ---------------------------------------------------------------------------------------

def _axis_basis(n, lo, hi):
    """Eigenvectors V (columns), V^-1 and eigenvalues of [1, -2, 1] with the axis' faces."""
    N = n + 1
    nodes = np.arange(0 if lo == "N" else 1, n + (1 if hi == "D" else 2))
    if lo == hi:
        num, den, modes = 1, N, nodes
    else:
        num, den, modes = 1, 2 * N, 2 * np.arange(1, N + 1) - 1
    # angle = pi * (node * mode) / den, the integer product reduced mod 2 den first
    arg = np.pi * ((np.outer(nodes, modes) * num) % (2 * den)) / den
    V = np.sin(arg) if lo == "D" else np.cos(arg)
    w = np.ones(len(nodes))
    w[nodes == 0] = 0.5
    w[nodes == N] = 0.5
    wm = np.ones(len(modes))
    if lo == hi == "N":
        wm[[0, -1]] = 0.5
    W = (2.0 / N) * wm[:, None] * V.T * w[None, :]
    lam = -4 * np.sin(np.pi * modes / (2 * den)) ** 2
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return t(V), t(W), t(lam)


def _planes(x, M, axis):
    """M applied along axis 1 (y) or 2 (x) of a complex [z, y, x] field."""
    M = M.to(torch.complex128)
    return x @ M.T if axis == 2 else torch.matmul(M, x)


def _tridiag(sub, diag, sup, x):
    """Thomas along the first axis; sub, diag, sup are functions of the row."""
    m = x.shape[0]
    cp, y = [None] * m, torch.empty_like(x)
    prev = None
    for l in range(m):
        d = diag(l) if l == 0 else diag(l) - sub(l) * cp[l - 1]
        cp[l] = sup(l) / d
        y[l] = x[l] / d if l == 0 else (x[l] - sub(l) * prev) / d
        prev = y[l]
    for l in range(m - 2, -1, -1):
        y[l] -= cp[l] * y[l + 1]
    return y


def _scheme(k, h):
    kh2 = (k * h) ** 2
    cf = 1 - kh2 / 12 + kh2 * kh2 / 360
    ik = 1j * k
    mu3 = 1 / (1 + (2 * ik * h / 3) * (1 + 2 * kh2 / 15))
    mu1 = (ik * h / 90 + (1 + kh2 / 30) / (6 * mu3)) / (1 + 2 * ik * h / 3)
    return dict(a=(1 + kh2 / 30) / 6, b=1 / 30, kappa=kh2 * cf, cf=cf, kh2=kh2, mu1=mu1, mu3=mu3,
                e1=np.exp(ik * h), e2=np.exp(2 * ik * h), p=mu1 + (2 * ik * h / 3) * (1 / 60 - mu1),
                q=1 - 2 * ik * h / 3 - 4 * ik * kh2 * h / 45, r=(4 * ik * h / 3) * (1 + 2 * kh2 / 15),
                s=(4 * ik * h / 3) * (1 / 60 - mu1))


def _direct(n, k, faces, F, order):
    """A u = F (order 6) or A_p u = F (order 2) solved mode by mode: with Dirichlet or Neumann
    x and y faces both operators are tridiagonal in z on the axes' eigenvectors."""
    h = 1.0 / (n + 1)
    Vx, Wx, lx = _axis_basis(n, faces[0], faces[1])
    Vy, Wy, ly = _axis_basis(n, faces[2], faces[3])
    X = _planes(_planes(F, Wx, 2), Wy, 1)
    sxy = (ly[:, None] + lx[None, :]).to(torch.complex128)
    pxy = (ly[:, None] * lx[None, :]).to(torch.complex128)
    c = _scheme(k, h)
    m = F.shape[0]
    if order == 6:
        off = 1 + c["a"] * sxy + c["b"] * pxy
        cen = -2 * off + sxy + c["a"] * pxy + c["kappa"]
        g0 = c["e1"] * c["mu3"] * (c["r"] - c["s"] * sxy)
        g1 = c["e2"] * c["mu3"] * (c["p"] * sxy + pxy / (30 * c["mu3"]) + c["q"])
    else:
        off = torch.ones_like(sxy)
        cen = sxy - 2 + c["kh2"]
        g0 = torch.full_like(sxy, 2j * k * h)  # U_-1 = U_1 + 2ikh U_0
        g1 = off
    one = [faces[4], faces[5]]

    def edge(l):
        return 0 if l == 0 else 1 if l == m - 1 else None

    def diag(l):
        e = edge(l)
        return cen + g0 if e is not None and one[e] == "S" else cen

    def inward(e):
        return off if one[e] == "D" else 2 * off if one[e] == "N" else off + g1

    def sup(l):
        return torch.zeros_like(off) if l == m - 1 else inward(0) if l == 0 else off

    def sub(l):
        return inward(1) if l == m - 1 else off

    U = _tridiag(sub, diag, sup, X)
    return _planes(_planes(U, Vy, 1), Vx, 2)


def _pad(x, dim, lo, hi):
    """One ghost layer per side along dim: even reflection at N, zero otherwise."""
    n = x.shape[dim]
    a = x.narrow(dim, 1, 1) if lo == "N" else torch.zeros_like(x.narrow(dim, 0, 1))
    b = x.narrow(dim, n - 2, 1) if hi == "N" else torch.zeros_like(x.narrow(dim, 0, 1))
    return torch.cat([a, x, b], dim)


def _d2(x, dim):
    n = x.shape[dim] - 2
    return x.narrow(dim, 2, n) - 2 * x.narrow(dim, 1, n) + x.narrow(dim, 0, n)


def _mid(x, *dims):
    for d in dims:
        x = x.narrow(d, 1, x.shape[d] - 2)
    return x


def _operator(n, k, faces, u):
    c = _scheme(k, 1.0 / (n + 1))
    P = _pad(_pad(_pad(u, 2, faces[0], faces[1]), 1, faces[2], faces[3]), 0, faces[4], faces[5])
    Dx, Dy, Dz = _d2(P, 2), _d2(P, 1), _d2(P, 0)
    Dxy, Dxz, Dyz = _d2(Dx, 1), _d2(Dx, 0), _d2(Dy, 0)
    out = _mid(Dx, 0, 1) + _mid(Dy, 0, 2) + _mid(Dz, 1, 2)
    out = out + c["a"] * (_mid(Dxy, 0) + _mid(Dxz, 1) + _mid(Dyz, 2)) + c["b"] * _d2(Dxy, 0) + c["kappa"] * u
    for side, row, p0, p1 in ((4, 0, 1, 2), (5, -1, -2, -3)):
        if faces[side] == "S":
            L = lambda q: _mid(_d2(q, 1), 0) + _mid(_d2(q, 0), 1)
            g1 = c["e2"] * c["mu3"] * (c["p"] * L(P[p1]) + _d2(_d2(P[p1], 1), 0) / (30 * c["mu3"])
                                       + c["q"] * _mid(P[p1], 0, 1))
            g0 = c["e1"] * c["mu3"] * (c["r"] * _mid(P[p0], 0, 1) - c["s"] * L(P[p0]))
            out[row] += g1 + g0
    return out


def _compact_rhs(n, k, faces, src, noise):
    """Compact right side of Gaussian sources, face terms of Neumann and radiating faces included."""
    h = 1.0 / (n + 1)
    c = _scheme(k, h)
    tabs = []
    for a in range(3):
        nodes = inputs.axis_nodes(n, faces[2 * a], faces[2 * a + 1]) * h
        t = (nodes[None, :] - src.centers[:, a:a + 1]) / src.sigma
        e = np.exp(-0.5 * t * t)
        he = [np.ones_like(t), t, t * t - 1, t ** 3 - 3 * t, t ** 4 - 6 * t * t + 3]
        tabs.append([torch.from_numpy((-1 / src.sigma) ** q * he[q] * e).cuda() for q in range(5)])
    amps = torch.from_numpy(src.amps).cuda()

    def f(ox, oy, oz, cut=None):
        X, Y, Z = tabs[0][ox], tabs[1][oy], tabs[2][oz]
        if cut is not None:
            ax, i = cut
            X, Y, Z = [t[:, i:i + 1] if a == ax else t for a, t in enumerate((X, Y, Z))]
        out = torch.zeros((Z.shape[1], Y.shape[1], X.shape[1]), dtype=torch.complex128, device="cuda")
        for s in range(len(amps)):
            out += (amps[s] * Z[s])[:, None, None] * (Y[s][:, None] * X[s][None, :])[None]
        return out

    F = c["cf"] * f(0, 0, 0) + (h * h / 12) * (1 - c["kh2"] / 30) * (f(2, 0, 0) + f(0, 2, 0) + f(0, 0, 2))
    F += h ** 4 / 360 * (f(4, 0, 0) + f(0, 4, 0) + f(0, 0, 4)) + h ** 4 / 90 * (f(2, 2, 0) + f(2, 0, 2) + f(0, 2, 2))
    if noise is not None:
        F += c["cf"] * noise
    F *= h * h
    ik = 1j * k
    for a in range(3):
        for side in range(2):
            kind = faces[2 * a + side]
            if kind == "D":
                continue
            i = 0 if side == 0 else F.shape[2 - a] - 1
            sg = 1 if side == 0 else -1
            t1, t2 = [b for b in range(3) if b != a]

            def d(on, o1, o2):
                o = [0, 0, 0]
                o[a], o[t1], o[t2] = on, o1, o2
                return (sg if on & 1 else 1) * f(*o, cut=(a, i))

            if kind == "N":
                term = (-(h ** 3 / 3) * (1 - c["kh2"] / 20) * d(1, 0, 0) - h ** 5 / 60 * d(3, 0, 0)
                        - 7 * h ** 5 / 180 * (d(1, 2, 0) + d(1, 0, 2)))
            else:
                f0, f1, f2 = d(0, 0, 0), d(1, 0, 0), d(2, 0, 0)
                b1 = ik * f0 + f1
                b2 = ik * ik * f0 + 2 * ik * f1 + f2
                b3 = ik ** 3 * f0 + 3 * ik * ik * f1 + 3 * ik * f2 + d(3, 0, 0)
                bt = ik * d(0, 2, 0) + d(1, 2, 0) + ik * d(0, 0, 2) + d(1, 0, 2)
                Fb = (h * h / 6 + k * k * h ** 4 / 45) * b1 - ik * h ** 4 / 90 * b2 + h ** 4 / 120 * (b3 - bt)
                term = -c["e1"] * c["mu3"] * (2 * h * Fb + c["mu1"] * h ** 5 / 3 * bt)
            F.narrow(2 - a, i, 1).sub_(term)
    return F


def _exact_gradient(case, seed):
    st = prepare(case, seed)
    theta = torch.from_numpy(st["trainer"].params()).cuda().double().requires_grad_(True)
    x = st["x"].double()
    st["trainer"].close()
    a, o = x.permute(0, 4, 1, 2, 3), 0
    chans = (2, 16, 16, 16, 2)
    for l in range(4):
        ci, co = chans[l], chans[l + 1]
        W = theta[o:o + co * ci * 27].view(co, ci, 3, 3, 3)
        b = theta[o + co * ci * 27:o + co * ci * 27 + co]
        o += co * ci * 27 + co
        P = torch.nn.functional.pad(a, (1, 1, 1, 1, 1, 1))
        m = a.shape[2:]
        out = b.view(1, co, 1, 1, 1)
        for t in range(27):
            dz, dy, dx = t // 9, t // 3 % 3, t % 3
            v = P[:, :, dz:dz + m[0], dy:dy + m[1], dx:dx + m[2]]
            out = out + torch.einsum("oc,bczyx->bozyx", W[:, :, dz, dy, dx], v)
        a = torch.nn.functional.gelu(out) if l < 3 else out
    y = torch.complex(a[:, 0], a[:, 1])
    c = _scheme(case["kh"], 1.0)
    Dx, Dy, Dz = _d2(y, 3), _d2(y, 2), _d2(y, 1)
    Dxy, Dxz, Dyz = _d2(Dx, 2), _d2(Dx, 1), _d2(Dy, 1)
    op = (_mid(Dx, 1, 2) + _mid(Dy, 1, 3) + _mid(Dz, 2, 3) + c["a"] * (_mid(Dxy, 1) + _mid(Dxz, 2) + _mid(Dyz, 3))
          + c["b"] * _d2(Dxy, 1) + c["kappa"] * _mid(y, 1, 2, 3))
    res = op - _mid(torch.complex(x[..., 0], x[..., 1]), 1, 2, 3)
    loss = (res.real ** 2 + res.imag ** 2).sum() / (2 * res.numel())
    loss.backward()
    return dict(loss=float(loss.detach()), grad=theta.grad.detach())


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        return _exact_gradient(case, seed)
    if kind == "batch":
        us = []
        for p in _problems(case):
            F = _compact_rhs(p["n"], p["k"], p["faces"], _batch_sources(p, seed), None)
            us.append(_direct(p["n"], p["k"], p["faces"], F, 6))
        return dict(u=us, rc=None)
    n, k, faces = case["n"], complex(case["kr"], case["ki"]), case["faces"]
    mx, my, mz = _dims(n, faces)
    shape = (mz, my, mx)
    if kind == "pinv":
        return _direct(n, k, faces, _field(shape, seed), 2)
    if kind == "apply":
        return _operator(n, k, faces, _field(shape, seed))
    if kind == "residual":
        r = _field(shape, seed) - _operator(n, k, faces, _field(shape, seed + 1))
        return dict(r=r, sumsq=torch.view_as_real(r).square().sum().reshape(1))
    F = _compact_rhs(n, k, faces, _sources(case, seed), _noise(case, seed, shape))
    return F if kind == "rhs" else dict(u=_direct(n, k, faces, F, 6), rc=None)
