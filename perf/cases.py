"""The calls that this library's performance is judged by, each through its public entry points.

A case is one call that a simulation makes: a backward-Euler heat run, a Helmholtz or Poisson solve, a
batch of independent solves, a Navier-Stokes projection step, a grain-growth step, or a differentiable
heat run with its backward pass. Every axis is a power of two (the library takes no other), so odd shapes
are unequal axes, and odd counts are numbers of steps, problems and order parameters.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  the device fields and solver contexts that a program holds before the call
    run(state)           one call; returns the fields that it computes
    work(case)           bytes and operations that the call cannot do without
    exact(case, seed)    the same outputs from eigenvector expansions or conjugate gradients in float64
"""
from __future__ import annotations

import math

import torch

import paper_2510_11152_gb300 as fas

TOL = 1e-10  # relative residual of every solve, the library's default


def listed():
    return [
        # the smallest heat run: latency and launches
        dict(name="heat2d_128_f64", kind="heat", nx=128, ny=128, nz=1, prec="f64", bc="neumann", steps=10, dt=1e-3,
             source=False, inner=1),
        # an everyday mixed-precision run whose levels all fit in the L2 cache
        dict(name="heat2d_1024_mixed", kind="heat", nx=1024, ny=1024, nz=1, prec="mixed", bc="neumann", steps=10,
             dt=1e-3, source=True, inner=1),
        # the benchmark's grid and parameters, fewer steps
        dict(name="heat2d_8192_mixed", kind="heat", nx=8192, ny=8192, nz=1, prec="mixed", bc="neumann", steps=3,
             dt=1e-4, source=True, inner=2),
        # the default precision on a large grid with unequal axes and both boundary kinds
        dict(name="heat2d_4096x2048_f64", kind="heat", nx=4096, ny=2048, nz=1, prec="f64", bc="xdir", steps=3,
             dt=1e-4, source=True, inner=1),
        # the paper's Dirichlet problem (its convergence test) at 1024^2, default precision
        dict(name="dirichlet2d_1024_f64", kind="solve", nx=1024, ny=1024, nz=1, prec="f64", bc="dirichlet", alpha=1.0,
             beta=1.0, inner=1),
        # the large 3D heat run of the benchmark, one step
        dict(name="heat3d_512_mixed", kind="heat", nx=512, ny=512, nz=512, prec="mixed", bc="neumann", steps=1,
             dt=1e-4, source=False, inner=3),
        # 3D at the default precision, unequal axes
        dict(name="heat3d_256x128x64_f64", kind="heat", nx=256, ny=128, nz=64, prec="f64", bc="dirichlet", steps=2,
             dt=1e-3, source=True, inner=1),
        # many independent solves of unequal sizes in one launch
        dict(name="batch96_2048_mixed", kind="batch", count=96, nmax=2048, prec="mixed", inner=1),
        # the 3D lid-driven cavity, first-order scheme, default precision
        dict(name="ns3d_128_f64", kind="ns", dim=3, n=128, order=1, prec="f64", inner=1),
        # a 2D flow, second-order scheme, mixed precision
        dict(name="ns2d_512_mixed", kind="ns", dim=2, n=512, order=2, prec="mixed", inner=1),
        # the paper's grain-growth grid with part of its order parameters (periodic solves)
        dict(name="grain_512_q128_mixed", kind="grain", nx=512, ny=512, nz=1, q=128, prec="mixed", inner=1),
        # training through the heat run: forward and backward, per-cell diffusivity, default precision
        dict(name="adjoint_512_f64", kind="adjoint", nx=512, ny=512, nz=1, steps=10, dt=1e-3, prec="f64", inner=1),
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo, hi)


def draw(rng):
    kind = rng.choice(["heat", "heat", "heat", "solve", "batch", "ns", "grain", "adjoint"])
    prec, inner = rng.choice([("f64", 1), ("mixed", 1), ("mixed", 2)])
    if kind in ("heat", "solve"):
        dim = rng.choice([2, 2, 3])
        k = rng.randint(6, 13 if prec == "mixed" else 12) if dim == 2 else rng.randint(5, 8)
        axes = [1 << max(4, k - rng.choice([0, 0, 1, 2])) for _ in range(dim)]
        c = dict(kind=kind, nx=axes[0], ny=axes[1], nz=axes[2] if dim == 3 else 1, prec=prec)
        cells = c["nx"] * c["ny"] * c["nz"]
        if kind == "heat":
            most = 10 if cells <= 1 << 20 else (4 if cells <= 1 << 23 else 2)
            c |= dict(bc=rng.choice(["neumann", "neumann", "dirichlet", "xdir", "periodic"]),
                      steps=rng.randint(1, most), dt=round(10 ** rng.uniform(-4, -3), 7), source=rng.random() < 0.5)
        else:
            c |= dict(bc="dirichlet", alpha=rng.choice([0.0, 1.0]), beta=1.0)
    elif kind == "batch":
        c = dict(kind=kind, count=rng.randint(3, 96), nmax=_pow2(rng, 7, 11), prec=prec)
    elif kind == "ns":
        dim = rng.choice([2, 3])
        c = dict(kind=kind, dim=dim, n=_pow2(rng, 6, 10) if dim == 2 else _pow2(rng, 5, 7), order=rng.choice([1, 2]),
                 prec=prec)
    elif kind == "grain":
        n = _pow2(rng, 6, 9)
        c = dict(kind=kind, nx=n, ny=n >> rng.choice([0, 0, 1]), nz=1, q=int(round(2 ** rng.uniform(2, 7))), prec=prec)
    else:
        n = _pow2(rng, 6, 9)
        c = dict(kind=kind, nx=n, ny=n >> rng.choice([0, 0, 1]), nz=1, steps=rng.randint(2, 10),
                 dt=round(10 ** rng.uniform(-4, -3), 7), prec=prec)
    c["inner"] = inner
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

def _shape(c):
    return (c["ny"], c["nx"]) if c["nz"] == 1 else (c["nz"], c["ny"], c["nx"])


def _gen(seed, k=0):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + k) % (1 << 62))


def _rand(g, *n):
    return torch.rand(*n, dtype=torch.float64, device="cuda", generator=g)


def _axes(shape):
    h = 1.0 / max(shape)
    return [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * h for n in shape]


def _outer(vs):
    out = vs[0]
    for v in vs[1:]:
        out = out.unsqueeze(-1) * v
    return out


def _noisy_cos(shape, g):
    """The slowest cosine mode plus 1e-2 of uniform noise (the heat runs' initial field)."""
    u = _rand(g, *shape).mul_(2e-2).sub_(1e-2)
    return u.add_(_outer([torch.cos(math.pi * x) for x in _axes(shape)]))


def _gaussians(shape, g, count, sigma, lo=-1.0, hi=1.0):
    """Sum of Gaussian bumps with random centres and amplitudes."""
    r = _rand(g, count, len(shape) + 1)
    cen, amp = r[:, :-1], lo + (hi - lo) * r[:, -1]
    f = [torch.exp(-((x[None] - cen[:, a:a + 1]) ** 2) / (2 * sigma * sigma)) for a, x in enumerate(_axes(shape))]
    if len(shape) == 2:
        return (f[0] * amp[:, None]).t() @ f[1]
    return torch.einsum("kz,ky,kx->zyx", f[0] * amp[:, None], f[1], f[2])


def _smoothed_normal(n, g):
    """N(0,1) smoothed by three damped-Jacobi averages (the batch's right-hand sides)."""
    f = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    for _ in range(3):
        p = torch.nn.functional.pad(f[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
        f = 0.5 * f + 0.125 * (p[:-2, 1:-1] + p[2:, 1:-1] + p[1:-1, :-2] + p[1:-1, 2:])
    return f


def _bc(c, dim):
    kind = {"neumann": 0, "dirichlet": 1, "periodic": 2, "xdir": 0}[c["bc"]]
    bc = [kind] * 6
    if c["bc"] == "xdir":  # Dirichlet on the x faces, Neumann on the others
        bc[0] = bc[1] = 1
    return bc[:2 * dim]


def _precision(c):
    return fas.FAS_MIXED if c["prec"] == "mixed" else fas.FAS_FP64


def _problems(c, seed):
    """The batch's problems: sizes from 64 up to nmax, diffusivities in [0.5, 2], two time steps."""
    r = torch.rand(c["count"], 3, dtype=torch.float64, generator=torch.Generator().manual_seed(int(seed) + 17)).tolist()
    sizes = [n for n in (64, 128, 256, 512, 1024, 2048) if n <= c["nmax"]]
    # the share of each size is fixed, so that another seed is as much work
    return [dict(n=sizes[k % len(sizes)], kappa=0.5 + 1.5 * r[k][1], dt=1e-4 if r[k][2] < 0.5 else 1e-3)
            for k in range(c["count"])]


_NS = dict(Re=100.0, dt=1e-3, lid=(1.0, 0.0, 0.0))


def _inputs(c, seed):
    g = _gen(seed)
    kind = c["kind"]
    if kind == "heat":
        s = _shape(c)
        return dict(u0=_noisy_cos(s, g), f=_gaussians(s, g, 16, 0.02 if len(s) == 2 else 0.1) if c["source"] else None)
    if kind == "solve":  # f of p = prod sin(pi sin(pi x)) under the operator, plus bumps that differ by seed
        s = _shape(c)
        p = _outer([torch.sin(math.pi * torch.sin(math.pi * x)) for x in _axes(s)])
        return dict(f=_gaussians(s, g, 8, 0.05).mul_(10.0).add_(p, alpha=20.0))
    if kind == "batch":
        return dict(f=[_smoothed_normal(p["n"], g) for p in _problems(c, seed)])
    if kind == "ns":
        s = (c["n"],) * c["dim"]
        out = {}
        for a, nm in enumerate("UVW"[:c["dim"]]):
            for when in ("_old", "_new"):
                if when == "_new" and c["order"] == 1:
                    v = torch.zeros(s, dtype=torch.float64, device="cuda")
                elif when == "_new":  # u^n of the second-order scheme, near u^{n-1}
                    v = out[nm + "_old"] + 1e-2 * _gaussians(s, g, 6, 0.15)
                else:
                    v = 0.5 * _gaussians(s, g, 6, 0.15)
                v.select(c["dim"] - 1 - a, c["n"] - 1).zero_()  # the far wall's slot
                out[nm + when] = v
        out["P_old"] = 0.1 * _gaussians(s, g, 4, 0.2)
        out["P_new"] = torch.zeros(s, dtype=torch.float64, device="cuda")
        return out
    if kind == "grain":
        s = _shape(c)
        return dict(eta0=_rand(g, c["q"], *s).mul_(2e-3).sub_(1e-3))
    if kind == "adjoint":
        s = _shape(c)
        return dict(u0=_noisy_cos(s, g), f=_gaussians(s, g, 16, 0.05),
                    kappa=1.0 + 0.5 * torch.tanh(_gaussians(s, g, 8, 0.1, -2.0, 2.0)),
                    target=_gaussians(s, g, 4, 0.15))
    raise ValueError(kind)


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = dict(case=c, **_inputs(c, seed))
    kw = dict(precision=_precision(c), inner_cycles=c["inner"], kmax=60, tol=TOL)
    if kind == "heat":
        s = _shape(c)
        st["solver"] = fas.Solver(s, 1.0 / max(s), alpha=1.0, beta=c["dt"], bc=_bc(c, len(s)), **kw)
        st["u"] = torch.empty_like(st["u0"])
    elif kind == "solve":
        s = _shape(c)
        st["solver"] = fas.Solver(s, 1.0 / max(s), alpha=c["alpha"], beta=c["beta"], bc=_bc(c, len(s)), **kw)
        st["u"] = torch.empty_like(st["f"])
    elif kind == "batch":
        probs = _problems(c, seed)
        st["ctxs"] = [fas.fas_create(fas.make_params((p["n"], p["n"]), 1.0 / p["n"], alpha=1.0, beta=p["dt"],
                                                     kappa_const=p["kappa"], **kw)) for p in probs]
        st["all"] = torch.empty(sum(p["n"] ** 2 for p in probs), dtype=torch.float64, device="cuda")
        st["u"] = [v.view(p["n"], p["n"]) for v, p in zip(st["all"].split([p["n"] ** 2 for p in probs]), probs)]
    elif kind == "ns":
        sp, pp = fas.fas_default_params(), fas.fas_default_params()
        for p in (sp, pp):
            p.precision, p.inner_cycles, p.kmax, p.coarsest, p.tol = kw["precision"], c["inner"], 60, 4, TOL
        pp.coarse_exact = 1
        st["ns"] = fas.ns_create((c["n"],) * c["dim"], 1.0 / c["n"], _NS["Re"], _NS["dt"], lid=_NS["lid"],
                                 order=c["order"], solver=sp, pressure=pp)
        names = [k for k in fas.NS_FIELDS if k in st]
        st["start"] = {k: st.pop(k) for k in names}
        st["fields"] = {k: torch.empty_like(v) for k, v in st["start"].items()}
    elif kind == "grain":
        sp = fas.fas_default_params()
        sp.precision, sp.inner_cycles, sp.kmax, sp.tol = kw["precision"], c["inner"], 60, TOL
        st["gg"] = fas.gg_create(_shape(c), 2.0, 0.25, c["q"], solver=sp)
        st["eta"] = torch.empty_like(st["eta0"])
    else:
        for k in ("u0", "f", "kappa"):
            st[k].requires_grad_(True)
        st["options"] = kw
    return st


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "heat":  # a run from its initial field, in place
        u = state["u"].copy_(state["u0"])
        state["solver"].heat_run(u, state["f"], c["dt"], c["steps"])
        return u
    if kind == "solve":
        u = state["u"].zero_()
        state["solver"].solve(u, state["f"])
        return u
    if kind == "batch":
        state["all"].zero_()
        fas.fas_solve_batched(state["ctxs"], state["u"], state["f"])
        return state["all"]
    if kind == "ns":  # one step from the same flow
        for k, v in state["fields"].items():
            v.copy_(state["start"][k])
        fas.ns_projection_step(state["ns"], state["fields"])
        return state["fields"]
    if kind == "grain":
        eta = state["eta"].copy_(state["eta0"])
        fas.gg_step(state["gg"], eta)
        return eta
    for k in ("u0", "f", "kappa"):
        state[k].grad = None
    n = max(_shape(c))
    uT = fas.HeatSolve.apply(state["u0"], state["f"], state["kappa"], 1.0 / n, c["dt"], c["steps"], 10, state["options"])
    loss = ((uT - state["target"]) ** 2).sum()
    loss.backward()
    return dict(uT=uT.detach(), g_u0=state["u0"].grad, g_f=state["f"].grad, g_kappa=state["kappa"].grad)


def work(case):
    """Bytes: every input field read once, every output field written once. Operations: six cycles of
    four sweeps and a residual on all levels for each solve, which is about what reaches TOL."""
    c, kind = case, case["kind"]

    def solves(cells, dim, count):
        return count * cells * 2 ** dim / (2 ** dim - 1) * 6 * 5 * (2 * dim + 2)

    if kind == "batch":
        cells = sum(p["n"] ** 2 for p in _problems(c, 0))
        return dict(bytes=16 * cells, flops=solves(cells, 2, 1))
    if kind == "ns":
        cells, d = c["n"] ** c["dim"], c["dim"]
        fields_in = d + 1 if c["order"] == 1 else 2 * d + 1
        return dict(bytes=8 * cells * (fields_in + 2 * d + 2), flops=solves(cells, d, d + 1))
    cells = c["nx"] * c["ny"] * c["nz"]
    dim = 2 if c["nz"] == 1 else 3
    if kind == "grain":
        return dict(bytes=16 * cells * c["q"], flops=solves(cells, dim, c["q"]))
    if kind == "adjoint":
        return dict(bytes=8 * cells * 8, flops=solves(cells, dim, 2 * c["steps"]))
    if kind == "solve":
        return dict(bytes=16 * cells, flops=solves(cells, dim, 1))
    return dict(bytes=8 * cells * (3 if c["source"] else 2), flops=solves(cells, dim, c["steps"]))


# ---------------------------------------------------------------------------------------------
# the same outputs in plain torch, float64
# ---------------------------------------------------------------------------------------------

def _modes(n, kind):
    """Orthonormal eigenvectors (rows) of the 1D second difference and -h^2 times their eigenvalues.
    neumann / dirichlet: cell-centred with mirrored / sign-changed ghosts; wall: faces between zeros."""
    i = torch.arange(n, device="cuda")
    if kind == "wall":
        k = torch.arange(1, n, device="cuda")
        v = torch.sin(math.pi / n * ((k[:, None] * k[None]) % (2 * n)).double()) * math.sqrt(2.0 / n)
    elif kind == "neumann":
        k = i
        v = torch.cos(math.pi / (2 * n) * ((k[:, None] * (2 * i + 1)[None]) % (4 * n)).double()) * math.sqrt(2.0 / n)
        v[0] /= math.sqrt(2.0)
    else:
        k = i + 1
        v = torch.sin(math.pi / (2 * n) * ((k[:, None] * (2 * i + 1)[None]) % (4 * n)).double()) * math.sqrt(2.0 / n)
        v[-1] /= math.sqrt(2.0)
    return v, 4.0 * torch.sin(math.pi / (2 * n) * k.double()) ** 2


def _along(m, x, axis):
    return torch.movedim(torch.tensordot(m, x, dims=([1], [axis])), 0, axis)


class _Spectral:
    """alpha u - beta Lap u on a box, diagonal in the products of 1D eigenvectors."""

    def __init__(self, kinds, shape, h, alpha, beta):
        self.periodic = kinds[0] == "periodic"
        lam = 0.0
        if self.periodic:
            for a, n in enumerate(shape):
                k = torch.arange(n if a < len(shape) - 1 else n // 2 + 1, device="cuda").double()
                w = 4.0 * torch.sin(math.pi / n * k) ** 2
                lam = w if a == 0 else lam.unsqueeze(-1) + w
            self.shape = shape
        else:
            self.v = []
            for a, (n, kd) in enumerate(zip(shape, kinds)):
                v, w = _modes(n, kd)
                self.v.append(v)
                lam = w if a == 0 else lam.unsqueeze(-1) + w
        self.diag = alpha + beta / (h * h) * lam
        self.zero = alpha == 0.0 and all(k in ("neumann", "periodic") for k in kinds)
        if self.zero:
            self.diag.reshape(-1)[0] = 1.0

    def to(self, x):
        if self.periodic:
            return torch.fft.rfftn(x, dim=tuple(range(x.ndim - len(self.shape), x.ndim)))
        for a, v in enumerate(self.v):
            x = _along(v, x, a)
        return x

    def back(self, x):
        if self.periodic:
            return torch.fft.irfftn(x, s=self.shape, dim=tuple(range(x.ndim - len(self.shape), x.ndim)))
        for a, v in enumerate(self.v):
            x = _along(v.t(), x, a)
        return x

    def solve(self, f):
        y = self.to(f) / self.diag
        if self.zero:
            y.reshape(-1)[0] = 0.0
        return self.back(y)


def _kinds(c, dim):
    return ["neumann"] * (dim - 1) + ["dirichlet"] if c["bc"] == "xdir" else [c["bc"]] * dim


def _cat(ax, *xs):
    return torch.cat(xs, dim=ax)


def _weno(a, b, c):
    """Third-order WENO value from three first differences, upwind side first."""
    b0, b1 = (b - a) ** 2, (c - b) ** 2
    w0, w1 = (1.0 / 3.0) / (1e-6 + b0) ** 2, (2.0 / 3.0) / (1e-6 + b1) ** 2
    return (w0 * 0.5 * (3.0 * b - a) + w1 * 0.5 * (b + c)) / (w0 + w1)


def _faces(x, ax):
    return _cat(ax, torch.zeros_like(x.narrow(ax, 0, 1)), x)


def _derivatives(phi, ax, h, normal, g_lo, g_hi):
    """Left- and right-biased WENO3 derivatives along axis ax (wall slot: 0)."""
    core = _faces(phi, ax) if normal else phi
    n = core.shape[ax]
    if normal:
        lo, hi = -core.narrow(ax, 1, 2).flip(ax), -core.narrow(ax, n - 3, 2).flip(ax)
    else:
        lo, hi = 2 * g_lo - core.narrow(ax, 0, 2).flip(ax), 2 * g_hi - core.narrow(ax, n - 2, 2).flip(ax)
    ext = _cat(ax, lo, core, hi)
    d = torch.diff(ext, dim=ax) / h
    start, count = (1, n - 2) if normal else (0, n)
    v = [d.narrow(ax, start + k, count) for k in range(4)]
    dm, dp = _weno(v[0], v[1], v[2]), _weno(v[3], v[2], v[1])
    if normal:
        pad = torch.zeros_like(phi.narrow(ax, 0, 1))
        dm, dp = _cat(ax, dm, pad), _cat(ax, dp, pad)
    return dm, dp


def _convection(phi, advect, comp, h, lid):
    dim = phi.ndim
    fc = dim - 1 - comp
    out = torch.zeros_like(phi)
    for a in range(dim):
        ax = dim - 1 - a
        dm, dp = _derivatives(phi, ax, h, a == comp, 0.0, lid[comp] if a == dim - 1 else 0.0)
        if a == comp:
            adv = phi
        else:
            ph = _faces(advect[a], ax)
            s = 0.5 * (ph.narrow(ax, 0, phi.shape[ax]) + ph.narrow(ax, 1, phi.shape[ax]))
            t = 0.5 * (s.narrow(fc, 0, phi.shape[fc] - 1) + s.narrow(fc, 1, phi.shape[fc] - 1))
            adv = _cat(fc, t, torch.zeros_like(t.narrow(fc, 0, 1)))
        out += torch.where(adv > 0, adv * dm, adv * dp)
    out.select(fc, phi.shape[fc] - 1).zero_()
    return out


def _gradient(p, comp, h):
    fc = p.ndim - 1 - comp
    return _cat(fc, torch.diff(p, dim=fc) / h, torch.zeros_like(p.narrow(fc, 0, 1)))


def _face_laplacian(u, comp, h):
    out = torch.zeros_like(u)
    for ax in range(u.ndim):
        if ax == u.ndim - 1 - comp:
            lap = torch.diff(_faces(u, ax), n=2, dim=ax)
            out += _cat(ax, lap, torch.zeros_like(u.narrow(ax, 0, 1)))
        else:
            m = u.shape[ax]
            out += torch.diff(_cat(ax, -u.narrow(ax, 0, 1), u, -u.narrow(ax, m - 1, 1)), n=2, dim=ax)
    return out / (h * h)


def _exact_ns(c, seed):
    dim, n, order = c["dim"], c["n"], c["order"]
    s, h, dt, lid = (n,) * dim, 1.0 / n, _NS["dt"], _NS["lid"]
    F = _inputs(c, seed)
    names = "UVW"[:dim]
    beta = dt / (_NS["Re"] * order)
    old = [F[m + "_old"] for m in names]
    cur = [F[m + "_new"] for m in names] if order == 2 else old
    tilde = []
    for comp in range(dim):
        fc = dim - 1 - comp
        if order == 1:
            phi, advect = cur[comp], cur
        else:
            phi = 0.5 * (3.0 * cur[comp] - old[comp])
            advect = [0.5 * (cur[a] + tilde[a]) if a < comp else 0.5 * (3.0 * cur[a] - old[a]) for a in range(dim)]
        f = cur[comp] - dt * _convection(phi, advect, comp, h, lid) - dt * _gradient(F["P_old"], comp, h)
        if order == 2:
            f += beta * _face_laplacian(cur[comp], comp, h)
        if comp != dim - 1:  # the moving wall, once for each implicit or explicit part
            f.select(0, n - 1).add_(order * 2.0 * beta * lid[comp] / (h * h))
        kinds = ["dirichlet"] * dim
        kinds[fc] = "wall"
        x = _Spectral(kinds, s, h, 1.0, beta).solve(f.narrow(fc, 0, n - 1))
        tilde.append(_cat(fc, x, torch.zeros_like(x.narrow(fc, 0, 1))))
    div = sum(torch.diff(_faces(tilde[a], dim - 1 - a), dim=dim - 1 - a) for a in range(dim)) / h
    p = _Spectral(["neumann"] * dim, s, h, 0.0, dt).solve(-div)
    out = dict(P_new=p, P_old=F["P_old"] + p)
    for a, m in enumerate(names):
        new = tilde[a] - dt * _gradient(p, a, h)
        out[m + "_old"], out[m + "_new"] = (new, tilde[a]) if order == 1 else (cur[a], new)
    return out


def _kappa_operator(kappa, h, dt):
    """u -> u - dt div(kappa grad u), homogeneous Neumann, face values the mean of two cells."""
    wy, wx = 0.5 * (kappa[1:] + kappa[:-1]), 0.5 * (kappa[:, 1:] + kappa[:, :-1])

    def apply(u):
        gy, gx = wy * torch.diff(u, dim=0), wx * torch.diff(u, dim=1)
        z = torch.nn.functional.pad
        div = z(gy, (0, 0, 0, 1)) - z(gy, (0, 0, 1, 0)) + z(gx, (0, 1)) - z(gx, (1, 0))
        return u - dt / (h * h) * div
    return apply


def _cg(apply, b, x):
    """Conjugate gradients to 1e-14 of b (checked now and then, to leave the GPU queue full)."""
    r = b - apply(x)
    p, rr, stop = r.clone(), (r * r).sum(), 1e-28 * float((b * b).sum())
    for it in range(5000):
        q = apply(p)
        al = rr / (p * q).sum()
        x, r = x + al * p, r - al * q
        new = (r * r).sum()
        if it % 32 == 31 and float(new) <= stop:
            break
        p, rr = r + new / rr * p, new
    return x


def _exact_adjoint(c, seed):
    I = _inputs(c, seed)
    h, dt = 1.0 / max(_shape(c)), c["dt"]
    A = _kappa_operator(I["kappa"], h, dt)
    us = [I["u0"]]
    for _ in range(c["steps"]):
        us.append(_cg(A, us[-1] + dt * I["f"], us[-1]))
    lam = 2.0 * (us[-1] - I["target"])
    g_f, kap = torch.zeros_like(lam), I["kappa"].clone().requires_grad_(True)
    g_k = torch.zeros_like(lam)
    for n in range(c["steps"], 0, -1):
        lam = _cg(A, lam, lam)
        g_f += dt * lam
        g_k -= torch.autograd.grad((lam * _kappa_operator(kap, h, dt)(us[n])).sum(), kap)[0]
    return dict(uT=us[-1], g_u0=lam, g_f=g_f, g_kappa=g_k)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "heat":
        s = _shape(c)
        I = _inputs(c, seed)
        S = _Spectral(_kinds(c, len(s)), s, 1.0 / max(s), 1.0, c["dt"])
        y = S.to(I["u0"])
        f = S.to(I["f"]) if I["f"] is not None else None
        del I
        for _ in range(c["steps"]):
            if f is not None:
                y = y.add_(f, alpha=c["dt"])
            y = y.div_(S.diag)
        return S.back(y)
    if kind == "solve":
        s = _shape(c)
        return _Spectral(_kinds(c, len(s)), s, 1.0 / max(s), c["alpha"], c["beta"]).solve(_inputs(c, seed)["f"])
    if kind == "batch":
        F = _inputs(c, seed)["f"]
        return torch.cat([_Spectral(["neumann"] * 2, f.shape, 1.0 / p["n"], 1.0, p["dt"] * p["kappa"]).solve(f).reshape(-1)
                          for p, f in zip(_problems(c, seed), F)])
    if kind == "ns":
        return _exact_ns(c, seed)
    if kind == "grain":  # the model's constants: 1, 1, 1, 1, 2
        e = _inputs(c, seed)["eta0"]
        phi = (e * e).sum(0)
        rhs = e - 0.25 * (-e + e ** 3 + 2.0 * e * (phi - e * e))
        return _Spectral(["periodic"] * 2, _shape(c), 2.0, 1.0, 0.25 * 2.0).solve(rhs)
    return _exact_adjoint(c, seed)
