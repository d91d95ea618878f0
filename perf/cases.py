"""What is measured: the calls a user's program makes, over the range of their sizes.

A case is a dict of plain values; its "kind" says which call one pass is:

  loop      five free-boundary steps (levelset_advance, init_domain, step), the
            last with reinitialisation: one cycle of the time loop every
            free-boundary program runs ("shape": disc, star, twoball, ellipsoid4)
  levelset  one levelset_advance with reinitialisation
  etd       two ETD steps on a fixed domain ("scheme" picks the integrator)
  phi       one phi_combination on given vectors
  adjoint   the torch wrapper's trajectory, forward and backward
  poisson   one Poisson solve with a node-field beta

Inputs are drawn on the GPU from the seed.  `exact` evaluates the same
quantities with dense FP64 torch arrays: the embedded-boundary operator and
the level-set step as their formulas state them, the phi functions by
Chebyshev expansion (no Krylov tolerance), the Poisson solution by conjugate
gradients to the rounding level, gradients by torch's differentiation.
"""
import math

import numpy as np
import torch

from paper_2209_15095_gb300 import autograd, etd

F64 = torch.float64
BAND = 6.0
TOL = {"disc": 1e-8, "star": 1e-7, "twoball": 1e-5, "ellipsoid4": 1e-5}


def listed():
    return [
        # the smallest program: a 2D front on 64^2, all launches and waits
        {"name": "disc2d-64-loop", "kind": "loop", "shape": "disc", "n": 64, "precision": "fp64"},
        # the main configuration in both precisions: a 3D star-shaped front
        {"name": "star3d-128-loop", "kind": "loop", "shape": "star", "n": 128, "precision": "fp64"},
        {"name": "star3d-128-mixed-loop", "kind": "loop", "shape": "star", "n": 128, "precision": "mixed"},
        # two competing species, each with its own front, on the largest free-boundary grid
        {"name": "twoball3d-256-mixed-loop", "kind": "loop", "shape": "twoball", "n": 256, "precision": "mixed"},
        # four space dimensions
        {"name": "ellipsoid4d-48-mixed-loop", "kind": "loop", "shape": "ellipsoid4", "n": 48, "precision": "mixed"},
        # the level set alone on an odd grid whose rows are not whole words
        {"name": "levelset3d-193", "kind": "levelset", "n": 193, "precision": "fp64"},
        # ETD2 on a large fixed domain: the largest grid in mixed precision, an FP64 one
        {"name": "etd2-ball-512-mixed", "kind": "etd", "ndim": 3, "n": 512, "precision": "mixed", "scheme": "etd2"},
        {"name": "etd2-ball-384", "kind": "etd", "ndim": 3, "n": 384, "precision": "fp64", "scheme": "etd2"},
        # a Runge-Kutta integrator on a medium domain: four launches a step, phi_3
        {"name": "etd4rk-ball-101", "kind": "etd", "ndim": 3, "n": 101, "precision": "fp64", "scheme": "etd4rk"},
        # the phi-function combination by itself, 2D, an odd size
        {"name": "phi-disc-1001", "kind": "phi", "ndim": 2, "n": 1001, "precision": "fp64"},
        # training through the solver: forward and backward with a node-field beta
        {"name": "adjoint-ball-128", "kind": "adjoint", "n": 128, "steps": 10, "precision": "fp64"},
        # the steady problem on the virus-shaped domain
        {"name": "poisson-virus-321", "kind": "poisson", "n": 321},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["loop", "loop", "loop", "levelset", "etd", "etd", "phi", "adjoint", "poisson"])
    precision = rng.choice(["fp64", "mixed"])
    if kind == "loop":
        shape = rng.choice(["disc", "star", "twoball", "ellipsoid4"])
        lo, hi = {"disc": (48, 640), "star": (64, 192), "twoball": (112, 224), "ellipsoid4": (30, 46)}[shape]
        return {"kind": kind, "shape": shape, "n": _log(rng, lo, hi), "precision": precision}
    if kind == "levelset":
        return {"kind": kind, "n": _log(rng, 64, 240), "precision": precision}
    if kind == "etd":
        ndim = rng.choice([2, 3, 3, 4])
        scheme = rng.choice(["etd2", "etd2", "etd1", "etd2rk", "etd3", "etd3rk", "etd4rk"])
        many = scheme in ("etd2rk", "etd3rk", "etd4rk")
        lo, hi = {2: (100, 1000 if many else 2000), 3: (56, 220 if many else 380), 4: (24, 48 if many else 64)}[ndim]
        return {"kind": kind, "ndim": ndim, "n": _log(rng, lo, hi), "precision": precision, "scheme": scheme}
    if kind == "phi":
        ndim = rng.choice([2, 3])
        return {"kind": kind, "ndim": ndim, "n": _log(rng, *{2: (100, 2000), 3: (56, 320)}[ndim]),
                "precision": precision}
    if kind == "adjoint":
        return {"kind": kind, "n": _log(rng, 40, 128), "steps": rng.randint(4, 10), "precision": precision}
    return {"kind": "poisson", "n": _log(rng, 81, 480)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _axes(n, lo, hi, ndim):
    """The node coordinates along each axis, shaped to broadcast over the grid."""
    ax = lo + (hi - lo) / (n - 1) * torch.arange(n, dtype=F64, device="cuda")
    return [ax.view([n if e == d else 1 for e in range(ndim)]) for d in range(ndim)]


def _angular(xs, r, g, degree):
    """A random polynomial of degree <= `degree` of the unit direction, max|Y| = 1."""
    rs = torch.where(r > 0, r, torch.ones_like(r))
    un = [x / rs for x in xs]
    Y = torch.zeros_like(r)
    for _ in range(degree * 3):
        t = 2.0 * torch.rand((), generator=g, dtype=F64, device="cuda") - 1.0
        for _ in range(int(torch.randint(1, degree + 1, (), generator=g, device="cuda"))):
            a = torch.randn(len(xs), generator=g, dtype=F64, device="cuda")
            t = t * sum(a[d] * un[d] for d in range(len(xs)))
        Y = Y + t
    return Y / Y.abs().max()


def _smooth_noise(shape, g, sweeps=3):
    U = torch.rand(shape, generator=g, dtype=F64, device="cuda")
    for _ in range(sweeps):
        m = sum(U.roll(s, d) for d in range(U.ndim) for s in (-1, 1)) / (2 * U.ndim)
        U = U + (2.0 / 3.0) * (m - U)
    return U


def _problem(case, seed):
    """Grid, initial fields and parameters of a case: {"n", "lo", "hi", "h", "phi", "u",
    "beta", "mu", "reaction", "rparams", "dt", "tol", "m_max"}."""
    g = _gen(seed)
    kind, n = case["kind"], case["n"]
    jit = 1.0 + 0.02 * (torch.rand(8, generator=g, dtype=F64, device="cuda").cpu().numpy() - 0.5)
    p = {"mu": (1.0, 1.0), "beta": (1.0, 1.0), "reaction": "logistic", "rparams": (), "dt": 5e-3, "m_max": 40}
    shape = case.get("shape", {"levelset": "star"}.get(kind, "ball"))
    ndim = {"disc": 2, "star": 3, "twoball": 3, "ellipsoid4": 4}.get(shape, case.get("ndim", 3))
    box = {"disc": 4.0, "star": 6.0, "twoball": 8.0, "ellipsoid4": 5.0}.get(shape, {2: 1.0, 3: 8.0, 4: 5.0}[ndim])
    if kind == "adjoint":
        box = 6.0
    if kind == "poisson":
        ndim, box = 2, 1.0
    xs = _axes(n, -box, box, ndim)
    r = torch.sqrt(sum(x * x for x in xs))
    if kind == "poisson":
        # the virus-shaped domain: x = (a + b sin 12t) cos t, y = (a + b/2 sin 12t) sin t
        t = np.linspace(0.0, 2.0 * math.pi, 200001)
        cx = (0.6 * jit[0] + 0.1 * np.sin(12 * t)) * np.cos(t)
        cy = (0.6 * jit[0] + 0.05 * np.sin(12 * t)) * np.sin(t)
        psi = np.unwrap(np.arctan2(cy, cx))
        ang = np.arctan2(np.broadcast_to(xs[1].cpu().numpy(), (n, n)), np.broadcast_to(xs[0].cpu().numpy(), (n, n)))
        R = np.interp(np.mod(ang - psi[0], 2.0 * math.pi) + psi[0], psi, np.hypot(cx, cy))
        p["phi"] = [r - torch.tensor(R, dtype=F64, device="cuda")]
        c = 1.0 + torch.rand(3, generator=g, dtype=F64, device="cuda")
        p["field"] = (2.0 + torch.sin(c[0] * xs[0] * xs[1])).contiguous()
        p["source"] = (torch.exp(c[1] * xs[0]) * torch.cos(c[2] * xs[1])).contiguous()
        p["u"] = [torch.zeros_like(r)]
        p["tol"] = 1e-12
    elif shape == "disc":
        R = 1.0 * jit[0]
        p["phi"] = [r - R]
        p["u"] = [torch.cos(math.pi * r / (2 * R)) * (0.9 + 0.1 * _angular([x.expand_as(r) for x in xs], r, g, 3))]
        p["mu"], p["dt"], p["m_max"] = (2.0, 2.0), 1e-2, 30
    elif shape == "star":
        r0 = 1.5 * (1.0 + 0.2 * _angular([x.expand_as(r) for x in xs], r, g, 4))
        p["phi"] = [r - r0]
        p["u"] = [(1.0 - r / r0) * (0.5 + 0.5 * _smooth_noise(tuple(r.shape), g))]
    elif shape == "twoball":
        p["phi"], p["u"] = [], []
        for s, cx in enumerate((-2.0, 2.0)):
            rc = torch.sqrt((xs[0] - cx * jit[s]) ** 2 + xs[1] ** 2 + xs[2] ** 2)
            p["phi"].append(rc - 1.5 * jit[2 + s])
            p["u"].append(torch.cos(math.pi * rc / (3.0 * jit[2 + s])))
        p["beta"], p["mu"], p["reaction"], p["rparams"] = (1.0, 0.5), (1.0, 0.8), "competition", (0.5, 0.8, 1.2)
    elif shape == "ellipsoid4":
        a = [1.5 * jit[0], 1.2 * jit[1], jit[2], jit[3]]
        rho = torch.sqrt(sum((xs[d] / a[d]) ** 2 for d in range(4)))
        p["phi"] = [min(a) * (rho - 1.0)]
        p["u"] = [torch.cos(math.pi * rho / 2.0)]
    else:  # a fixed ball (disc) well inside the box
        R = (4.0 if kind == "adjoint" else {2: 0.85, 3: 7.0, 4: 3.0}[ndim]) * jit[0]
        p["phi"] = [r - R]
        m = torch.ones((), dtype=F64, device="cuda")
        for d in range(ndim):
            m = m * (1.0 + 0.2 * torch.cos((2.0 + d) * xs[d] * jit[1 + d] / R))
        p["u"] = [(0.7 * torch.cos(math.pi * r / (2 * R)) * m).contiguous()]
        p["dt"] = 1e-2 if ndim != 2 else 2e-4
    p["u"] = [torch.where(f < 0, u, torch.zeros_like(u)) for f, u in zip(p["phi"], p["u"])]
    if kind == "adjoint":
        # beta = 1 + 0.3 g, g smooth noise of correlation length 1 clipped to [-1, 1]
        k2 = sum(torch.fft.fftfreq(n, d=12.0 / (n - 1), dtype=F64, device="cuda").view(
            [n if e == d else 1 for e in range(3)]) ** 2 for d in range(3))
        w = torch.randn((n,) * 3, generator=g, dtype=F64, device="cuda")
        f = torch.fft.ifftn(torch.fft.fftn(w) * torch.exp(-math.pi ** 2 * k2)).real
        p["field"] = (1.0 + 0.3 * ((f - f.mean()) / f.std()).clamp(-1.0, 1.0)).contiguous()
        p["reaction"], p["rparams"] = "logistic_ak", (1.0, 1.0)
        p["alpha"] = 1.0 + 0.2 * float(jit[4] - 1.0)
        p["weights"] = _smooth_noise((n,) * 3, g)
    if "tol" not in p:
        p["tol"] = TOL.get(shape, 1e-8 if kind == "phi" else 1e-7)
        if shape == "star" and case["precision"] == "mixed":
            p["tol"] = 1e-5
    if kind == "phi":
        u = p["u"][0]
        p["v"] = [u, p["dt"] * u * (1.0 - u), p["dt"] * _smooth_noise(tuple(u.shape), g)]
    p.update(n=(n,) * ndim, lo=(-box,) * ndim, hi=(box,) * ndim, h=2.0 * box / (n - 1), ndim=ndim,
             prepare_reinit=shape in ("star", "ellipsoid4"))
    return p


def prepare(case, seed):
    p = _problem(case, seed)
    kind = case["kind"]
    ctx = etd.Context(p["n"], p["lo"], p["hi"], nspecies=len(p["phi"]), precision=case.get("precision", "fp64"),
                      tol=p["tol"], m_max=p["m_max"], reaction="none" if kind == "poisson" else p["reaction"],
                      rparams=p["rparams"], mu=p["mu"], beta=p["beta"], adjoint=kind == "adjoint",
                      scheme=case.get("scheme", "etd2"))
    s = {"kind": kind, "ctx": ctx, "dt": p["dt"], "phi0": p["phi"], "u0": p["u"]}
    if kind in ("loop", "levelset"):
        for f in p["phi"]:
            ctx.levelset_prepare(f, reinit=p["prepare_reinit"])
        s["phi"] = [torch.empty_like(f) for f in p["phi"]]
        s["u"] = [torch.empty_like(u) for u in p["u"]]
        for i, (f, u) in enumerate(zip(p["phi"], p["u"])):
            # u is given on the domain of the prepared level set
            u.copy_(torch.where(f < 0, u, torch.zeros_like(u)))
            ctx.init_domain(i, f)
    elif kind == "etd":
        ctx.init_domain(0, p["phi"][0])
        s["u"] = [torch.empty_like(p["u"][0])]
    elif kind == "phi":
        ctx.init_domain(0, p["phi"][0])
        s["v"], s["y"] = p["v"], torch.zeros_like(p["u"][0])
    elif kind == "adjoint":
        s["beta"], s["weights"], s["steps"] = p["field"].requires_grad_(), p["weights"], case["steps"]
        s["alpha"] = torch.tensor(p["alpha"], dtype=F64, device="cuda", requires_grad=True)
        s["u0"] = [p["u"][0].requires_grad_()]
    elif kind == "poisson":
        ctx.init_domain(0, p["phi"][0], p["field"])
        s["f"], s["u"], s["field"] = p["source"], [torch.empty_like(p["u"][0])], p["field"]
    ctx.sync()
    return s


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "loop":
        # a time loop started from the prepared fields (the context keeps F of
        # its last step as F_{n-1}, as in a program's own loop)
        for i in range(len(s["phi"])):
            s["phi"][i].copy_(s["phi0"][i])
            s["u"][i].copy_(s["u0"][i])
            ctx.init_domain(i, s["phi"][i])
        for k in range(5):
            for i in range(len(s["phi"])):
                ctx.levelset_advance(i, s["phi"][i], s["u"][i], s["dt"], k == 4)
            for i in range(len(s["phi"])):
                ctx.init_domain(i, s["phi"][i])
            ctx.step(s["dt"], s["u"])
        return {"phi": s["phi"], "u": s["u"]}
    if kind == "levelset":
        s["phi"][0].copy_(s["phi0"][0])
        s["u"][0].copy_(s["u0"][0])
        ctx.levelset_advance(0, s["phi"][0], s["u"][0], s["dt"], True)
        return {"phi": s["phi"], "u": s["u"]}
    if kind == "etd":
        s["u"][0].copy_(s["u0"][0])
        ctx.step(s["dt"], s["u"])
        ctx.step(s["dt"], s["u"])
        return {"u": s["u"]}
    if kind == "phi":
        ctx.phi_combination(0, s["dt"], *s["v"], s["y"])
        return {"y": s["y"]}
    if kind == "adjoint":
        u0, beta, alpha = s["u0"][0], s["beta"], s["alpha"]
        uT = autograd.trajectory(ctx, u0, beta, alpha, s["phi0"][0], s["dt"], s["steps"])
        loss = (s["weights"] * uT * uT).sum()
        gu, gb, ga = torch.autograd.grad(loss, (u0, beta, alpha))
        return {"u": uT.detach(), "grad_u0": gu, "grad_beta": gb, "grad_alpha": ga}
    s["u"][0].zero_()
    ctx.poisson_solve(0, s["f"], s["u"][0], tol=1e-12)
    return {"u": s["u"]}


def work(case):
    """Inputs read once and outputs written once per call; the arithmetic of
    the tube's WENO stages and of one matrix-vector product per Krylov vector
    (their number from the spectral radius, which grows it like a square root)."""
    kind, n = case["kind"], case["n"]
    if kind == "poisson":
        pts = 0.28 * n * n
        return {"bytes": 32.0 * pts, "flops": 5.0 * n * pts * 26}
    if kind in ("loop", "levelset"):
        shape = case.get("shape", "star")
        N = {"disc": 2, "star": 3, "twoball": 3, "ellipsoid4": 4}[shape]
        h = 2.0 * {"disc": 4.0, "star": 6.0, "twoball": 8.0, "ellipsoid4": 5.0}[shape] / (n - 1)
        R = {"disc": 1.0, "star": 1.5, "twoball": 1.5, "ellipsoid4": 1.15}[shape]
        ball = {2: math.pi, 3: 4 * math.pi / 3, 4: math.pi ** 2 / 2}[N]
        species = 2 if shape == "twoball" else 1
        inside = ball * (R / h) ** N
        tube = ball * ((R / h + 6.0) ** N - max(R / h - 6.0, 0.0) ** N)
        steps = 5 if kind == "loop" else 1
        stages = 3 * (steps + math.ceil(12 * math.sqrt(N)))
        dt = 1e-2 if shape == "disc" else 5e-3
        m = 10 + 1.5 * math.sqrt(4 * N * dt / h ** 2) if kind == "loop" else 0.0
        flops = tube * ((106 * N + 7) * stages + steps * 3 * math.ceil(12 * math.sqrt(N)) * (2 * N + 2))
        flops += steps * inside * m * (4 * N + 10)
        return {"bytes": species * steps * (16.0 * tube + 24.0 * inside), "flops": species * flops}
    N = case.get("ndim", 3)
    box, R = (6.0, 4.0) if kind == "adjoint" else {2: (1.0, 0.85), 3: (8.0, 7.0), 4: (5.0, 3.0)}[N]
    h = 2.0 * box / (n - 1)
    inside = {2: math.pi, 3: 4 * math.pi / 3, 4: math.pi ** 2 / 2}[N] * (R / h) ** N
    dt = 2e-4 if N == 2 else 1e-2
    m = 10 + 1.5 * math.sqrt(4 * N * dt / h ** 2)
    if kind == "phi":
        return {"bytes": 32.0 * inside, "flops": inside * m * (4 * N + 10)}
    if kind == "adjoint":
        return {"bytes": case["steps"] * 80.0 * inside, "flops": case["steps"] * inside * 5 * m * (4 * N + 10)}
    calls = 2 * {"etd2rk": 2, "etd3rk": 3, "etd4rk": 4}.get(case["scheme"], 1)
    return {"bytes": calls * 32.0 * inside, "flops": calls * inside * m * (4 * N + 10)}


# ------------------------------------------------------------------- exact
def _sh(a, d, s):
    """a at the node s steps along axis d, the edge value past the box."""
    n = a.shape[d]
    return a.index_select(d, (torch.arange(n, device=a.device) + s).clamp(0, n - 1))


class _Operator:
    """C of the embedded-boundary discretisation of div(beta grad u) on the
    computational points: ghost faces enter the diagonal with their clamped
    interpolation weights.  beta: a number or a node field."""

    def __init__(self, phi, h, lo, beta):
        N = phi.ndim
        inside = phi < 0
        comp = inside.clone()
        for d in range(N):
            comp &= _sh(inside, d, 1) & _sh(inside, d, -1)
        self.comp, self.N, self.h = comp, N, h
        self.m = comp.to(F64)
        self.w = {}  # (d, s): ghost weight at the points with a ghost face there
        pts = comp.nonzero()
        grad = None
        for d in range(N):
            for s in (-1, 1):
                q = pts.clone()
                q[:, d] += s
                gi = (~comp[tuple(q.T)]).nonzero().ravel()
                if not len(gi):
                    self.w[d, s] = None
                    continue
                ip, iq = pts[gi], q[gi]
                ir = iq.clone()
                ir[:, d] += s
                fp, fq, fr = phi[tuple(ip.T)], phi[tuple(iq.T)], phi[tuple(ir.T)]
                th = fq / (fq - fr)
                w = th / (1.0 + th)
                c3 = (fr < 0).nonzero().ravel()
                if len(c3):
                    def grad(i):
                        out = []
                        for e in range(N):
                            a, b = i.clone(), i.clone()
                            a[:, e] += 1
                            b[:, e] -= 1
                            out.append((phi[tuple(a.T)] - phi[tuple(b.T)]) / (2.0 * h))
                        return torch.stack(out, -1)

                    w[c3] = self._case3(ip[c3], iq[c3], fp[c3], fq[c3], grad(ip[c3]), grad(iq[c3]), lo)
                self.w[d, s] = (tuple(ip.T), w.clamp(0.0, 1.0))
        self.set_beta(beta)

    def _case3(self, ip, iq, fp, fq, gp, gq, lo):
        h, N = self.h, self.N
        xp, xq = lo + h * ip.to(F64), lo + h * iq.to(F64)
        G1 = xq - (fq / (gq * gq).sum(-1))[:, None] * gq
        G2 = xp - (fp / (gp * gp).sum(-1))[:, None] * gp
        if N == 2:  # affine interpolation through x_p, G1, G2
            e1, e2, e = G1 - xp, G2 - xp, xq - xp
            det = e1[:, 0] * e2[:, 1] - e1[:, 1] * e2[:, 0]
            bad = det.abs() < 1e-12 * h * h
            ds = torch.where(bad, torch.ones_like(det), det)
            c1 = (e[:, 0] * e2[:, 1] - e[:, 1] * e2[:, 0]) / ds
            c2 = (e1[:, 0] * e[:, 1] - e1[:, 1] * e[:, 0]) / ds
            return torch.where(bad, fq / fp, 1.0 - c1 - c2)
        nb = gq + gp  # the hyperplane through G1 and G2
        nb = nb / nb.norm(dim=-1, keepdim=True)
        t = G2 - G1
        tl = t.norm(dim=-1, keepdim=True)
        tt = torch.where(tl >= 1e-12 * h, t / tl.clamp_min(1e-300), torch.zeros_like(t))
        nn = nb - (nb * tt).sum(-1, keepdim=True) * tt
        nn = nn / nn.norm(dim=-1, keepdim=True)
        num, den = ((xq - G1) * nn).sum(-1), ((xp - G1) * nn).sum(-1)
        bad = den.abs() < 1e-12 * h
        return torch.where(bad, fq / fp, num / torch.where(bad, torch.ones_like(den), den))

    def set_beta(self, beta):
        """Face coefficients and diagonal (differentiable in a node field)."""
        node = isinstance(beta, torch.Tensor)
        self.face, D = {}, 0.0
        for (d, s), gw in self.w.items():
            f = 0.5 * (beta + beta.roll(-s, d)) if node else float(beta)
            k = torch.ones_like(self.m)
            if gw is not None:
                k[gw[0]] = 1.0 - gw[1]
            self.face[d, s] = f
            D = D + f * k
        self.D = D * self.m
        b = float(beta.max()) if node else float(beta)
        self.rho = 4.0 * self.N * b / self.h ** 2

    def __call__(self, x):
        """C x for x that is zero off the computational points."""
        acc = -self.D * x
        for (d, s), f in self.face.items():
            acc = acc + f * x.roll(-s, d)
        return acc * (self.m / self.h ** 2)


def _phi_k(k, z):
    """phi_k(z) = sum_i z^i / (i + k)!, on an array of non-positive numbers."""
    small = np.abs(z) < 1.0
    zs = np.where(small, z, 0.0)
    ser = sum(zs ** i / math.factorial(i + k) for i in range(24))
    zl = np.where(small, -1.0, z)
    f = np.exp(zl)
    for j in range(k):
        f = (f - 1.0 / math.factorial(j)) / zl
    return np.where(small, ser, f)


def _combination(C, dt, vs):
    """sum_k phi_k(dt C) v_k: Chebyshev expansions on [-rho, 0], one Clenshaw recurrence."""
    rho = dt * C.rho
    K = int(40 + 4.0 * math.sqrt(rho) + 0.15 * rho)
    th = math.pi * (np.arange(2 * K) + 0.5) / (2 * K)
    z = 0.5 * rho * (np.cos(th) - 1.0)
    cos = np.cos(np.outer(np.arange(K), th))
    co = [cos @ _phi_k(k, z) / K for k in range(len(vs))]
    vs = [v * C.m for v in vs]
    size = [max(float(v.abs().max()), 1e-300) for v in vs]
    top = max(size)
    used = [j for j in range(K) if any(abs(c[j]) * s > 1e-18 * top for c, s in zip(co, size))]
    b1 = b2 = torch.zeros_like(vs[0])
    for j in range(used[-1] if used else 0, -1, -1):
        d = sum(float(c[j]) * v for c, v in zip(co, vs))
        if j == 0:
            return 0.5 * d + (2.0 * dt / rho) * C(b1) + b1 - b2
        b1, b2 = d + 2.0 * ((2.0 * dt / rho) * C(b1) + b1) - b2, b1


def _reaction(p, us):
    if p["reaction"] == "competition":
        a, b, r = p["rparams"]
        return [us[0] * (1.0 - us[0] - a * us[1]), r * us[1] * (1.0 - us[1] - b * us[0])]
    al = p.get("alpha", 1.0)
    return [al * u * (1.0 - u) for u in us]


def _etd_steps(C, p, u, scheme, steps):
    dt = p["dt"]

    def F(x):
        return _reaction(p, [x])[0]

    z = torch.zeros_like(u)
    hist = []
    for _ in range(steps):
        f = F(u)
        hist = [f] + hist[:2]
        if scheme in ("etd2rk", "etd3rk", "etd4rk"):
            if scheme == "etd2rk":
                a = _combination(C, dt, [u, dt * f])
                u = a + _combination(C, dt, [z, z, dt * (F(a) - f)])
                continue
            a = _combination(C, 0.5 * dt, [u, 0.5 * dt * f])
            if scheme == "etd3rk":
                b = _combination(C, dt, [u, dt * (2.0 * F(a) - f)])
                v2, v3 = -3.0 * f + 4.0 * F(a) - F(b), 4.0 * f - 8.0 * F(a) + 4.0 * F(b)
            else:
                b = _combination(C, 0.5 * dt, [u, 0.5 * dt * F(a)])
                c = _combination(C, 0.5 * dt, [a, 0.5 * dt * (2.0 * F(b) - f)])
                ab = F(a) + F(b)
                v2, v3 = -3.0 * f + 2.0 * ab - F(c), 4.0 * f - 4.0 * ab + 4.0 * F(c)
            u = _combination(C, dt, [u, dt * f, dt * v2, dt * v3])
        elif scheme == "etd1" or len(hist) == 1:
            u = _combination(C, dt, [u, dt * f])
        elif scheme == "etd3" and len(hist) == 3:
            f1, f2 = hist[1:]
            u = _combination(C, dt, [u, dt * f, dt * (1.5 * f - 2.0 * f1 + 0.5 * f2), dt * (f - 2.0 * f1 + f2)])
        else:
            u = _combination(C, dt, [u, dt * f, dt * (f - hist[1])])
    return u


def _tube(phi, h):
    s = phi.abs() < BAND * h
    t = s.clone()
    for d in range(phi.ndim):
        t |= _sh(s, d, 1) | _sh(s, d, -1)
    return t


def _stencils(T, reach):
    """Flat indices of the nodes of T and of their neighbours along each axis."""
    n, at = T.shape, T.nonzero()
    st = [int(np.prod(n[d + 1:])) for d in range(T.ndim)]
    base = sum(at[:, d] * st[d] for d in range(T.ndim))
    nb = [[base + ((at[:, d] + k).clamp(0, n[d] - 1) - at[:, d]) * st[d] for k in range(-reach, reach + 1)]
          for d in range(T.ndim)]
    return at, base, nb


def _weno(v1, v2, v3, v4, v5):
    s1 = 13.0 / 12.0 * (v1 - 2.0 * v2 + v3) ** 2 + 0.25 * (v1 - 4.0 * v2 + 3.0 * v3) ** 2
    s2 = 13.0 / 12.0 * (v2 - 2.0 * v3 + v4) ** 2 + 0.25 * (v2 - v4) ** 2
    s3 = 13.0 / 12.0 * (v3 - 2.0 * v4 + v5) ** 2 + 0.25 * (3.0 * v3 - 4.0 * v4 + v5) ** 2
    a1, a2, a3 = 0.1 / (1e-6 + s1) ** 2, 0.6 / (1e-6 + s2) ** 2, 0.3 / (1e-6 + s3) ** 2
    return (a1 * (v1 / 3.0 - 7.0 * v2 / 6.0 + 11.0 * v3 / 6.0) + a2 * (-v2 / 6.0 + 5.0 * v3 / 6.0 + v4 / 3.0)
            + a3 * (v3 / 3.0 + 5.0 * v4 / 6.0 - v5 / 6.0)) / (a1 + a2 + a3)


def _rk3(phi, base, nb, h, dt, rate, positive):
    """One TVD-RK3 step of phi_t = rate(|grad phi|) on the nodes `base`."""
    def L(f):
        acc = 0.0
        for nd in nb:
            v = [f[i] for i in nd]
            q = [(v[k + 1] - v[k]) / h for k in range(6)]
            a, b = _weno(*q[:5]), _weno(*q[:0:-1])
            a, b = torch.where(positive, a, -a), torch.where(positive, b, -b)
            acc = acc + torch.maximum(a.clamp_min(0.0), -b.clamp_max(0.0)) ** 2
        return rate(torch.sqrt(acc))

    f0 = phi[base]
    f = phi.clone()
    f[base] = f0 + dt * L(phi)
    f[base] = 0.75 * f0 + 0.25 * (f[base] + dt * L(f))
    f[base] = f0 / 3.0 + 2.0 / 3.0 * (f[base] + dt * L(f))
    return f


def _reinit(phi, h):
    N, shape = phi.ndim, phi.shape
    _, base, nb = _stencils(_tube(phi, h), 3)
    f = phi.reshape(-1)
    S = f[base] / torch.sqrt(f[base] ** 2 + h * h)
    for _ in range(math.ceil(12.0 * math.sqrt(N))):
        f = _rk3(f, base, nb, h, 0.5 * h / math.sqrt(N), lambda g: S - S * g, S > 0)
    return f.reshape(shape).clamp(-BAND * h, BAND * h)


def _prepared(phi, h, reinit):
    phi = phi.clamp(-BAND * h, BAND * h)
    return _reinit(phi, h) if reinit else phi


def _advance(phi, u, h, lo, mu, dt, reinit):
    """One level-set step: (phi, extended u)."""
    N, shape, T = phi.ndim, phi.shape, _tube(phi, h)
    inside = phi < 0
    v = [inside.clone()]
    for d in range(N):
        v[0] &= _sh(inside, d, 1) & _sh(inside, d, -1)
    for k in range(2):
        v.append(v[k].clone())
        for d in range(N):
            v[k + 1] &= _sh(v[k], d, 1) & _sh(v[k], d, -1)
    n = [(_sh(phi, d, 1) - _sh(phi, d, -1)) / (2.0 * h) for d in range(N)]
    nrm = torch.sqrt(sum(x * x for x in n)).clamp_min(1e-12)
    n = [x / nrm for x in n]
    zero = torch.zeros_like(u)

    def along(q):
        return sum(n[d] * (_sh(q, d, 1) - _sh(q, d, -1)) for d in range(N)) / (2.0 * h)

    q0 = torch.where(v[0], u, zero)
    q1 = torch.where(v[1], along(q0), zero)
    q2 = torch.where(v[2], along(q1), zero)
    src = None
    for q, val in ((q2, v[2]), (q1, v[1]), (q0, v[0])):
        at, base, nb = _stencils(T & ~val, 1)
        q = q.reshape(-1).clone()
        nf = [x.reshape(-1)[base] for x in n]
        s = 0.0 if src is None else src[base]
        dtau = h / (2.0 * math.sqrt(N))
        for _ in range(math.ceil(12.0 * math.sqrt(N))):
            c = q[base]
            g = sum(nf[d] * torch.where(nf[d] > 0, c - q[nb[d][0]], q[nb[d][2]] - c) for d in range(N)) / h
            q[base] = c - dtau * (g - s)
        src = q
    ue = src
    at, base, nb = _stencils(T, 3)
    f = phi.reshape(-1)
    nf = [x.reshape(-1)[base] for x in n]
    st = [int(np.prod(shape[d + 1:])) for d in range(N)]
    us = []
    for k in (1.0, 2.0):
        i0, fr = [], []
        for d in range(N):
            s = (at[:, d].to(F64) - (f[base] + k * h) * nf[d] / h).clamp(0.0, shape[d] - 1.0)
            i0.append(torch.floor(s).to(torch.int64).clamp_max(shape[d] - 2))
            fr.append(s - i0[d])
        out = 0.0
        for corner in range(1 << N):
            w, q = 1.0, 0
            for d in range(N):
                bit = (corner >> d) & 1
                w = w * (fr[d] if bit else 1.0 - fr[d])
                q = q + (i0[d] + bit) * st[d]
            out = out + w * ue[q]
        us.append(out)
    V = mu * ((4.0 * us[0] - us[1]) / (2.0 * h)).clamp_min(0.0)
    nsub = max(1, math.ceil(dt * float(V.max()) * N / (0.5 * h)))
    yes = torch.ones_like(V, dtype=torch.bool)
    for _ in range(nsub):
        f = _rk3(f, base, nb, h, dt / nsub, lambda g: -V * g, yes)
    phi = f.reshape(shape).clamp(-BAND * h, BAND * h)
    return (_reinit(phi, h) if reinit else phi), ue.reshape(shape)


def exact(case, seed):
    p = _problem(case, seed)
    kind, h = case["kind"], p["h"]
    lo = torch.tensor(p["lo"], dtype=F64, device="cuda")
    if kind in ("loop", "levelset"):
        phi = [_prepared(f, h, p["prepare_reinit"]) for f in p["phi"]]
        u = [torch.where(f < 0, x, torch.zeros_like(x)) for f, x in zip(phi, p["u"])]
        if kind == "levelset":
            f, x = _advance(phi[0], u[0], h, lo, p["mu"][0], p["dt"], True)
            return {"phi": [f], "u": [x]}
        Fp = [None] * len(phi)
        for k in range(5):
            for i in range(len(phi)):
                phi[i], u[i] = _advance(phi[i], u[i], h, lo, p["mu"][i], p["dt"], k == 4)
            C = [_Operator(f, h, lo, p["beta"][i]) for i, f in enumerate(phi)]
            if len(phi) == 2:
                own = [torch.where(c.comp, x, torch.zeros_like(x)) for c, x in zip(C, u)]
                F = [_reaction(p, [u[0], own[1]])[0], _reaction(p, [own[0], u[1]])[1]]
            else:
                F = _reaction(p, u)
            for i, c in enumerate(C):
                f = F[i] * c.m
                fp = f if Fp[i] is None else torch.where(Fp[i][1] & c.comp, Fp[i][0], f)
                u[i] = _combination(c, p["dt"], [u[i], p["dt"] * f, p["dt"] * (f - fp)])
                Fp[i] = (f, c.comp)
        return {"phi": phi, "u": u}
    C = _Operator(p["phi"][0], h, lo, p.get("field", p["beta"][0]))
    if kind == "etd":
        return {"u": [_etd_steps(C, p, p["u"][0] * C.m, case["scheme"], 2)]}
    if kind == "phi":
        return {"y": _combination(C, p["dt"], p["v"])}
    if kind == "adjoint":
        beta, steps, dt = p["field"], case["steps"], p["dt"]

        def step(u, um, b, al):
            C.set_beta(b)
            f = al * u * (1.0 - u)
            fm = al * um * (1.0 - um)
            return _combination(C, dt, [u, dt * f, dt * (f - fm)])

        al = torch.tensor(p["alpha"], dtype=F64, device="cuda")
        us = [p["u"][0]]
        for k in range(steps):
            us.append(step(us[k], us[max(k - 1, 0)], beta, al))
        lam = [torch.zeros_like(x) for x in us]
        lam[steps] = 2.0 * p["weights"] * us[steps]
        gb, ga = torch.zeros_like(beta), torch.zeros_like(al)
        for k in range(steps - 1, -1, -1):
            with torch.enable_grad():
                x, xm = us[k].detach().requires_grad_(), us[max(k - 1, 0)].detach().requires_grad_()
                b, a = beta.detach().requires_grad_(), al.detach().requires_grad_()
                gx, gm, db, da = torch.autograd.grad(step(x, xm, b, a), (x, xm, b, a), lam[k + 1])
            lam[k] = lam[k] + gx
            lam[max(k - 1, 0)] = lam[max(k - 1, 0)] + gm
            gb, ga = gb + db, ga + da
        return {"u": us[steps], "grad_u0": lam[0], "grad_beta": gb, "grad_alpha": ga}
    # poisson: conjugate gradients on -C, restarted from the true residual
    f = p["source"] * C.m
    x = torch.zeros_like(f)
    for _ in range(4):
        r = C(x) - f
        d, rr = r.clone(), float((r * r).sum())
        stop = 1e-26 * float((f * f).sum())
        for _ in range(20 * case["n"]):
            q = -C(d)
            a = rr / float((d * q).sum())
            x = x + a * d
            r = r - a * q
            new = float((r * r).sum())
            d, rr = r + (new / rr) * d, new
            if rr < stop:
                break
    return {"u": [x]}
