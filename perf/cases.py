"""Performance cases: the calls a user of the solver makes, over the sizes and options it is used
with.

``listed()`` names them, ``draw(rng)`` gives one more of the same ranges, ``prepare`` builds what a
program holds before the call (inputs on the GPU, the solver handle), ``run`` is one pass through
the public entry points, ``work`` the bytes and operations the pass cannot do without, and
``exact`` the same outputs in float64 from plain torch: dense sine transforms, and time marching
(spectral for a constant a, conjugate gradients per step for a varying one).

A case is a dict of plain values.  ``kind`` says which call it stands for:
  solve      st_assemble_rhs + st_solve of one space-time system
  adjoint    autograd.heat_solve forward and backward (gradients in f, u0 and the nodal a)
  batch      BatchSolver.st_solve_batch over uneven instances
  prec       st_apply_prec (the float64 preconditioner of a float64 handle)
  prec32     st_apply_prec_f32 (the float32 preconditioner of a mixed handle)
  op         st_apply_op (the flipped operator Y T)
  gradients  st_assemble_rhs, st_grad_rhs and st_grad_a
"""
import math

import numpy as np
import torch

import paper_2201_10062_gb300 as P
from paper_2201_10062_gb300.autograd import heat_solve

DEV = "cuda"
F64 = torch.float64


def _case(name, kind, dim, mx, my, mz, n, scheme="theta", theta=1.0, coef="one", prec="PH",
          precision="mixed", tol=1e-8):
    return dict(name=name, kind=kind, dim=dim, mx=mx, my=my, mz=mz, n=n, scheme=scheme,
                theta=theta, coef=coef, prec=prec, precision=precision, tol=tol)


def listed():
    return [
        # the smallest solve: the 1D backward-Euler example, float64, bound by launches
        _case("solve_1d_fp64", "solve", 1, 63, 1, 1, 64, precision="fp64"),
        # the headline workload: 2D Crank-Nicolson, constant a, mixed precision
        _case("solve_cn2d_mixed", "solve", 2, 255, 255, 1, 256, theta=0.5),
        # the same in plain float64
        _case("solve_cn2d_fp64", "solve", 2, 255, 255, 1, 256, theta=0.5, precision="fp64"),
        # the largest grid of the configurations: 2D variable a, BDF2
        _case("solve_bdf2_511_mixed", "solve", 2, 511, 511, 1, 128, scheme="bdf2", coef="field"),
        # P_theta with a variable a (Chebyshev inner map), backward Euler
        _case("solve_ptheta_mixed", "solve", 2, 255, 255, 1, 128, coef="field", prec="Ptheta",
              tol=1e-10),
        # the 3D example of the paper, a small constant a given on the nodes
        _case("solve_3d_mixed", "solve", 3, 63, 63, 63, 64, coef="small", tol=1e-10),
        # inverse problems: forward and adjoint solve with all gradients, 100 time steps
        _case("adjoint_n100_mixed", "adjoint", 2, 127, 127, 1, 100, coef="field", tol=1e-10),
        # many uneven instances in one graph launch
        dict(name="batch_uneven", kind="batch", count=8, shapes=4, tol=1e-9),
        # the float32 preconditioner on an uneven grid with daily steps over a year
        _case("prec32_511x127_n365", "prec32", 2, 511, 127, 1, 365, theta=0.5, coef="field"),
        # the float64 preconditioner, 200 steps
        _case("prec64_127x255_n200", "prec", 2, 127, 255, 1, 200, coef="field",
              precision="fp64"),
        # the operator alone, as an outer iteration of the user's own applies it
        _case("op_255_n256", "op", 2, 255, 255, 1, 256, theta=0.5, coef="field",
              precision="fp64"),
        # right-hand side and gradient kernels around a solve
        _case("gradients_255_n128", "gradients", 2, 255, 255, 1, 128, theta=0.5, coef="field"),
    ]


_SMALLEST, _LARGEST = 3.0e4, 1.6e7  # unknowns of a drawn case


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "adjoint", "batch", "prec", "prec32",
                       "prec32", "op", "gradients"])
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 7), shapes=rng.randint(5, 10 ** 6),
                    tol=1e-9)
    most = 4.0e6 if kind == "adjoint" else _LARGEST
    dim = rng.choice([1, 2, 2, 2, 2, 3]) if kind in ("solve", "prec32", "prec", "op") else 2
    axis = {1: [255, 511, 1023], 2: [31, 63, 127, 255, 511], 3: [15, 31, 63]}[dim]
    while True:
        target = math.exp(rng.uniform(math.log(_SMALLEST), math.log(most)))
        mx = rng.choice(axis)
        my = rng.choice([a for a in axis if 1 / 8.5 <= a / mx <= 8.5]) if dim >= 2 else 1
        mz = rng.choice(axis) if dim == 3 else 1
        n = round(target / (mx * my * mz))
        if 8 <= n <= 520:
            break
    # half of the time axes are the powers of two that the paper uses, the others what came out
    if rng.random() < 0.5:
        n = 2 ** int(math.log2(n))
    scheme = rng.choice(["theta", "theta", "bdf2"])
    theta = rng.choice([0.5, 1.0]) if scheme == "theta" else 1.0
    coef = "field" if kind in ("adjoint", "gradients") else rng.choice(["one", "field"])
    precision = {"prec": "fp64", "prec32": "mixed"}.get(kind) or rng.choice(
        ["mixed", "mixed", "fp64"])
    prec = "PH"
    if kind == "solve" and precision == "mixed" and scheme == "theta" and rng.random() < 0.25:
        prec = "Ptheta"
    c = _case("", kind, dim, mx, my, mz, n, scheme, theta, coef, prec, precision,
              tol=1e-8 if precision == "fp64" and kind != "adjoint" else 1e-10)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _field(dim, mx, my, mz, seed):
    """Smooth nodal diffusion in [1/2, 3/2]: a seeded sum of sine modes, boundary nodes included."""
    r = np.random.default_rng(seed)
    k = np.arange(1, 9 if dim < 3 else 5)
    s = [np.sin(math.pi * np.outer(k, np.linspace(0.0, 1.0, len_ + 2))) for len_ in (mx, my, mz)]
    c = r.uniform(-1.0, 1.0, (len(k),) * dim)
    if dim == 1:
        f = c @ s[0]
    elif dim == 2:
        f = s[1].T @ c @ s[0]
    else:
        f = np.einsum("rqp,rk,qj,pi->kji", c, s[2], s[1], s[0], optimize=True)
    return np.ascontiguousarray(1.0 + 0.5 * f / np.abs(f).max())


def _nodal(c, seed):
    if c["coef"] == "one":
        return None
    if c["coef"] == "small":
        return np.full((c["mz"] + 2, c["my"] + 2, c["mx"] + 2), 1e-3)
    return _field(c["dim"], c["mx"], c["my"], c["mz"], seed)


def _spec(c, seed):
    return P.ProblemSpec(c["dim"], c["mx"], c["my"], c["n"], 1.0, c["scheme"], c["theta"],
                         _nodal(c, seed), c["prec"], c["precision"], mz=c["mz"])


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _modes(c):
    """The lowest sine mode on the interior grid, as one space vector."""
    s = [torch.sin(math.pi * torch.arange(1, k + 1, device=DEV, dtype=F64) / (k + 1))
         for k in (c["mx"], c["my"], c["mz"])]
    v = s[0]
    if c["dim"] >= 2:
        v = (s[1][:, None] * v[None, :]).reshape(-1)
    if c["dim"] == 3:
        v = (s[2][:, None] * v[None, :]).reshape(-1)
    return v


def _data(c, seed):
    """Forcing at t_0..t_n, initial value, u^(-1) (BDF2) and noise on the assembled system, shaped
    like the manufactured solution sin(pi x) sin(pi y) e^t."""
    g = _gen(seed)
    n, base = c["n"], _modes(c)
    amp = 1.0 + torch.rand(1, generator=g, device=DEV, dtype=F64)
    t = torch.arange(0, n + 1, device=DEV, dtype=F64) / n
    f = torch.exp(t)[:, None] * (amp * (1.0 + c["dim"] * math.pi ** 2) * base)[None, :]
    u0 = amp * base
    up = math.exp(-1.0 / n) * u0 if c["scheme"] == "bdf2" else None
    noise = 1e-3 * torch.randn(n, base.numel(), generator=g, device=DEV, dtype=F64)
    return f, u0, up, noise


def _observed(c, seed):
    """Forcing, initial value and noisy observations of the solution (a percent of the signal)."""
    f, u0, _, noise = _data(c, seed)
    t = torch.arange(1, c["n"] + 1, device=DEV, dtype=F64) / c["n"]
    return f, u0, torch.exp(t)[:, None] * u0[None, :] + 10.0 * noise


def _shapes(c):
    r = np.random.default_rng(c["shapes"])
    out = []
    for _ in range(c["count"]):
        mx, n = int(r.choice([63, 127, 255])), int(r.choice([32, 64, 128, 256, 512]))
        out.append(_case("", "solve", 2, mx, mx, 1, n, theta=float(r.choice([0.5, 1.0])),
                         coef="field", tol=c["tol"]))
    return out


def _seeds(c, seed):
    return [int(seed) * 131 + i for i in range(c["count"])]


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        shapes, seeds = _shapes(c), _seeds(c, seed)
        b = P.BatchSolver([_spec(s, q) for s, q in zip(shapes, seeds)])
        fH = []
        for i, (s, q) in enumerate(zip(shapes, seeds)):
            f, u0, up, noise = _data(s, q)
            fH.append(b.instance(i).st_assemble_rhs(f, u0, up, noise))
        return dict(case=c, batch=b, fH=fH)
    if kind == "adjoint":
        f, u0, obs = _observed(c, seed)
        a = torch.tensor(_nodal(c, seed), device=DEV, dtype=F64)
        spec = P.ProblemSpec(c["dim"], c["mx"], c["my"], c["n"], 1.0, c["scheme"], c["theta"],
                             None, c["prec"], c["precision"])
        return dict(case=c, spec=spec, f=f.requires_grad_(), u0=u0.requires_grad_(),
                    a=a.requires_grad_(), obs=obs)
    s = P.Solver(_spec(c, seed))
    if kind == "solve":
        f, u0, up, noise = _data(c, seed)
        return dict(case=c, solver=s, f=f, u0=u0, up=up, noise=noise)
    g = _gen(seed)
    v = torch.randn(c["n"], s.spec.m, generator=g, device=DEV, dtype=F64)
    if kind == "gradients":
        f, u0, up, noise = _data(c, seed)
        return dict(case=c, solver=s, f=f, u0=u0, up=up, noise=noise, lam=v, u=f[1:] + noise)
    return dict(case=c, solver=s, v=v)


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        outs, _ = state["batch"].st_solve_batch(state["fH"], tol=c["tol"])
        return outs
    if kind == "adjoint":
        u = heat_solve(state["f"], state["u0"], state["spec"], a_nodal=state["a"], tol=c["tol"])
        loss = 0.5 * (u - state["obs"]).square().sum()
        gf, gu0, ga = torch.autograd.grad(loss, (state["f"], state["u0"], state["a"]))
        return u.detach(), gf, gu0, ga
    s = state["solver"]
    if kind == "solve":
        fH = s.st_assemble_rhs(state["f"], state["u0"], state["up"], state["noise"])
        u, _ = s.st_solve(fH, tol=c["tol"])
        return u
    if kind == "prec":
        return s.st_apply_prec(state["v"])
    if kind == "prec32":
        return s.st_apply_prec_f32(state["v"])
    if kind == "op":
        return s.st_apply_op(state["v"])
    fH = s.st_assemble_rhs(state["f"], state["u0"], state["up"], state["noise"])
    gf, gu0, gup = s.st_grad_rhs(state["lam"])
    ga = s.st_grad_a(state["lam"], state["u"], state["u0"])
    return fH, gf, gu0, gup, ga


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        # the assembled right-hand sides and the fields in, the solutions out
        shapes = _shapes(c)
        return {"bytes": sum(16 * s["n"] * s["mx"] * s["my"] + 8 * (s["mx"] + 2) * (s["my"] + 2)
                             for s in shapes),
                "flops": sum(work(s)["flops"] for s in shapes)}
    m = c["mx"] * c["my"] * c["mz"]
    N = m * c["n"]
    nodes = (c["mx"] + 2) * (c["my"] + 2 if c["dim"] >= 2 else 1) * (
        c["mz"] + 2 if c["dim"] == 3 else 1)
    a = 0 if c["coef"] == "one" else 8 * nodes
    # one sine transform of length len along an axis by FFT, both ways along every axis
    lens = [c["n"], c["mx"], c["my"], c["mz"]]
    fft = sum(2 * 2.5 * math.log2(2 * (k + 1)) for k in lens if k > 1)
    sten = 4 * c["dim"] + 6
    if kind == "prec":
        return {"bytes": 16 * N, "flops": fft * N}
    if kind == "prec32":
        return {"bytes": 12 * N, "flops": fft * N}
    if kind == "op":
        return {"bytes": 16 * N + a, "flops": sten * N}
    if kind == "gradients":
        # rhs: f, noise in, f_H out; adjoint of it: lam in, gradient out; a: lam and u in
        return {"bytes": 8 * (3 * N + m) + 8 * (2 * N + m) + 16 * N + 2 * a,
                "flops": (3 + 2 + sten) * N}
    if kind == "adjoint":
        # f, u0, a, observations in; u and the three gradients out; two solves
        return {"bytes": 8 * (4 * N + 4 * m) + 2 * a, "flops": 2 * (fft + sten) * N}
    return {"bytes": 8 * (3 * N + 2 * m) + a, "flops": (fft + sten) * N}


# ------------------------------------------------------------------ float64 values, plain torch
def _sine(k):
    """The orthonormal DST-I matrix of order k."""
    i = torch.arange(1, k + 1, device=DEV, dtype=torch.int64)
    r = (i[:, None] * i[None, :]) % (2 * (k + 1))
    return math.sqrt(2.0 / (k + 1)) * torch.sin(math.pi * r.to(F64) / (k + 1))


class _Grid:
    """K = -div(a grad) on the interior nodes (face values are means of two nodes)."""

    def __init__(self, c, a):
        self.dim = c["dim"]
        self.len = [c["mx"], c["my"], c["mz"]][:self.dim]
        self.shape = tuple(reversed(self.len))
        one = torch.ones(tuple(k + 2 for k in self.shape), device=DEV, dtype=F64)
        self.a = one if a is None else a
        self.S = [_sine(k) for k in self.len]
        self.mu = []
        for k in self.len:
            i = torch.arange(1, k + 1, device=DEV, dtype=F64)
            self.mu.append(4.0 * torch.sin(0.5 * math.pi * i / (k + 1)).square() * (k + 1) ** 2)

    def face(self, ax):
        """Face values along axis ax (0 = x), on the interior lines."""
        d = self.dim - 1 - ax
        a = self.a
        for e in range(self.dim):
            if e != d:
                a = a.narrow(e, 1, a.shape[e] - 2)
        k = a.shape[d] - 1
        return 0.5 * (a.narrow(d, 0, k) + a.narrow(d, 1, k))

    def K(self, u):
        out = 0.0
        for ax in range(self.dim):
            pad = [0, 0] * ax + [1, 1]
            d = u.dim() - 1 - ax
            flux = self.face(ax) * torch.diff(torch.nn.functional.pad(u, pad), dim=d)
            out = out - torch.diff(flux, dim=d) * (self.len[ax] + 1) ** 2
        return out

    def dst(self, u):
        for ax in range(self.dim):
            u = torch.movedim(torch.movedim(u, -1 - ax, -1) @ self.S[ax], -1, -1 - ax)
        return u

    def eig(self, coef):
        """sum over the axes of coef[axis] times the a = 1 eigenvalues, on the spectral grid."""
        e = 0.0
        for ax in range(self.dim):
            e = e + (coef[ax] * self.mu[ax]).reshape((-1,) + (1,) * ax)
        return e


def _steps(g, c, b):
    """T u = b by time marching, block by block; b: (n, *grid)."""
    n, tau, th = c["n"], 1.0 / c["n"], c["theta"]
    bdf = c["scheme"] == "bdf2"
    d0, kc = (1.5, tau) if bdf else (1.0, th * tau)
    spread = float(g.a.max() - g.a.min())
    u = torch.empty_like(b)
    if spread == 0.0:  # one value of a: the sine transform diagonalises every block
        mu = g.eig([float(g.a.reshape(-1)[0])] * g.dim)
        v = g.dst(b)
        for k in range(n):
            r = v[k]
            if bdf:
                r = r + (2.0 * v[k - 1] if k > 0 else 0.0) - (0.5 * v[k - 2] if k > 1 else 0.0)
            elif k > 0:
                r = r + (1.0 - (1.0 - th) * tau * mu) * v[k - 1]
            v[k] = r / (d0 + kc * mu)
        return g.dst(v)
    mean = sum(float(g.face(ax).mean()) for ax in range(g.dim)) / g.dim
    inv = 1.0 / (d0 + kc * g.eig([mean] * g.dim))

    def A(x):
        return d0 * x + kc * g.K(x)

    zero = torch.zeros_like(b[0])
    for k in range(n):
        p1, p2 = (u[k - 1] if k > 0 else zero), (u[k - 2] if k > 1 else zero)
        if bdf:
            r = b[k] + 2.0 * p1 - 0.5 * p2
        else:
            r = b[k] + p1 - ((1.0 - th) * tau * g.K(p1) if th != 1.0 else 0.0)
        x = 2.0 * p1 - p2 if k > 1 else p1.clone()
        r = r - A(x)
        z = g.dst(g.dst(r) * inv)
        p, rz = z, (r * z).sum()
        for _ in range(24):  # the spectrum lies within a_max / a_min <= 3
            q = A(p)
            al = rz / ((p * q).sum() + 1e-300)
            x = x + al * p
            r = r - al * q
            z = g.dst(g.dst(r) * inv)
            rn = (r * z).sum()
            p = z + rn / (rz + 1e-300) * p
            rz = rn
        u[k] = x
    return u


def _rhs(g, c, f, u0, up, extra):
    n, tau, th = c["n"], 1.0 / c["n"], c["theta"]
    gr = lambda v: v.reshape(g.shape)  # noqa: E731
    if c["scheme"] == "bdf2":
        b = tau * f[1:]
        b[0] += 2.0 * u0 - 0.5 * (up if up is not None else u0)
        if n > 1:
            b[1] -= 0.5 * u0
    else:
        b = th * tau * f[1:] + (1.0 - th) * tau * f[:-1]
        b[0] += u0 - (1.0 - th) * tau * g.K(gr(u0)).reshape(-1)
    return b if extra is None else b + extra


def _T(g, c, u):
    n, tau, th = c["n"], 1.0 / c["n"], c["theta"]
    Ku = tau * g.K(u)
    if c["scheme"] == "bdf2":
        y = 1.5 * u + Ku
        y[1:] -= 2.0 * u[:-1]
        y[2:] += 0.5 * u[:-2]
    else:
        y = u + th * Ku
        y[1:] += (1.0 - th) * Ku[:-1] - u[:-1]
    return y


def _prec(g, c, v):
    """P_H^-1 v: the modulus of the symbol at each time frequency and eigenvalue of the averaged K."""
    n, tau, th = c["n"], 1.0 / c["n"], c["theta"]
    diag, off = 0.0, []
    for ax in range(g.dim):
        d = g.dim - 1 - ax
        f, h2 = g.face(ax), (g.len[ax] + 1) ** 2
        k = g.len[ax]
        diag = diag + (f.narrow(d, 0, k) + f.narrow(d, 1, k)).mean() * h2
        off.append(f.narrow(d, 1, k - 1).mean() * h2)
    # d - 2 sum e cos = (d - 2 sum e) + sum e mu0 h^2, with mu0 h^2 = 4 sin^2
    mu = diag - 2.0 * sum(off) + g.eig([o / (k + 1) ** 2 for o, k in zip(off, g.len)])
    x = math.pi * torch.arange(1, n + 1, device=DEV, dtype=F64) / (n + 1)
    x = x.reshape((n,) + (1,) * g.dim)
    e = torch.exp(1j * x)
    t = tau * mu
    if c["scheme"] == "bdf2":
        p = (1.5 + t - 2.0 * e + 0.5 * e * e).abs()
    else:
        p = ((1.0 + th * t) + ((1.0 - th) * t - 1.0) * e).abs()
    S = _sine(n)
    w = (S @ g.dst(v).reshape(n, -1)).reshape(v.shape) / p
    return g.dst((S @ w.reshape(n, -1)).reshape(v.shape))


def _tensor(a):
    return None if a is None else torch.tensor(a, device=DEV, dtype=F64)


def _exact_solve(c, seed):
    g = _Grid(c, _tensor(_nodal(c, seed)))
    b = _rhs(g, c, *_data(c, seed))
    return _steps(g, c, b.reshape((c["n"],) + g.shape)).reshape(c["n"], -1)


def _grad_a(g, c, lam, u, u0):
    """-tau sum_k lam_k^T (dK/da) (theta u_k + (1-theta) u_{k-1}) at the nodes."""
    n, tau, th = c["n"], 1.0 / c["n"], c["theta"]
    a = g.a.clone().requires_grad_()
    shape = (n,) + g.shape
    u, lam = u.reshape(shape), lam.reshape(shape)
    w = u if c["scheme"] == "bdf2" else th * u + (1.0 - th) * torch.cat(
        [u0.reshape((1,) + g.shape), u[:-1]])
    keep, g.a = g.a, a
    total = 0.0
    for ax in range(g.dim):
        pad = [0, 0] * ax + [1, 1]
        d = w.dim() - 1 - ax
        dw = torch.diff(torch.nn.functional.pad(w, pad), dim=d)
        dl = torch.diff(torch.nn.functional.pad(lam, pad), dim=d)
        total = total - tau * (g.len[ax] + 1) ** 2 * (g.face(ax) * (dw * dl).sum(0)).sum()
    g.a = keep
    return torch.autograd.grad(total, a)[0]


def _grad_rhs(g, c, lam):
    n, tau, th = c["n"], 1.0 / c["n"], c["theta"]
    gf = torch.zeros(n + 1, lam.shape[1], device=DEV, dtype=F64)
    if c["scheme"] == "bdf2":
        gf[1:] = tau * lam
        gu0 = 2.0 * lam[0] - (0.5 * lam[1] if n > 1 else 0.0)
        return gf, gu0, -0.5 * lam[0]
    gf[1:] += th * tau * lam
    gf[:-1] += (1.0 - th) * tau * lam
    gu0 = lam[0] - (1.0 - th) * tau * g.K(lam[0].reshape(g.shape)).reshape(-1)
    return gf, gu0, torch.zeros_like(gu0)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        return [_exact_solve(s, q) for s, q in zip(_shapes(c), _seeds(c, seed))]
    if kind == "solve":
        return _exact_solve(c, seed)
    g = _Grid(c, _tensor(_nodal(c, seed)))
    shape = (c["n"],) + g.shape
    if kind == "adjoint":
        f, u0, obs = _observed(c, seed)
        b = _rhs(g, c, f, u0, None, None)
        u = _steps(g, c, b.reshape(shape))
        # T^T lam = u - obs: the blocks are symmetric, so march backwards in time
        r = (u.reshape(c["n"], -1) - obs).reshape(shape)
        lam = _steps(g, c, torch.flip(r, (0,)))
        lam = torch.flip(lam, (0,)).reshape(c["n"], -1)
        u = u.reshape(c["n"], -1)
        gf, gu0, _ = _grad_rhs(g, c, lam)
        return u, gf, gu0, _grad_a(g, c, lam, u, u0)
    v = torch.randn(c["n"], math.prod(g.shape), generator=_gen(seed), device=DEV, dtype=F64)
    if kind in ("prec", "prec32"):
        return _prec(g, c, v.reshape(shape)).reshape(c["n"], -1)
    if kind == "op":
        return torch.flip(_T(g, c, v.reshape(shape)), (0,)).reshape(c["n"], -1)
    f, u0, up, noise = _data(c, seed)
    gf, gu0, gup = _grad_rhs(g, c, v)
    ga = _grad_a(g, c, v, f[1:] + noise, u0).reshape(-1)
    return _rhs(g, c, f, u0, up, noise), gf, gu0, gup, ga
