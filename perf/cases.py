"""The calls whose speed is measured: what a user of the library runs, at the sizes it is used at.

A case is one call, or one forward and one adjoint call, through the public entry points of
``paper_1810_11685_gb300``.  ``kind`` selects the call:

* ``prop``    H_a of a batch of initial pressures and H_a^* of a batch of sensor series (2D or 3D);
* ``grad``    the same through ``autograd.acoustic``: forward and backward;
* ``forward`` the whole opto-acoustic map mu -> fluence -> heating -> sensor series;
* ``jvp``     one Jacobian product of a Krylov iteration (fluence given);
* ``group``   Jacobian products on several grids at once (``Group.jvp``);
* ``da``      the fluence solve alone;
* ``medium``  the gradient in sound speed and density.

Grids are the interior plus ``pml`` nodes on every side.  Media are a water-like background with
elliptic inclusions, absorption maps a background with discs, sensors a ring or the perimeter, the time
step a CFL number times dx / c_max: the recipe of the repository's own workloads, made here on the GPU
from the seed alone.
"""
import math

import numpy as np
import torch

DEV = "cuda"
MM = 1e-3


# --------------------------------------------------------------------------------------------------
# the cases

def _case(name, kind, n, pml, *, batch=1, nt=0, prec="fp32", y=1.5, lossless=False, ns=128, dx=0.1, sensors="ring"):
    """n: interior extents, "nx,ny[,nz]" or one number for all of a 2D grid ("3d:n" of a 3D one)."""
    return dict(name=name, kind=kind, n=str(n), pml=pml, batch=batch, nt=nt, prec=prec, y=y, lossless=lossless, ns=ns,
                dx=dx, sensors=sensors)


def listed():
    return [
        # the smallest propagation a user waits for: one problem on the 128^2 grid of a 2D reconstruction study
        _case("2d-128-b1", "prop", 128, 20, nt=400, y=1.3),
        # the same grid in double precision, the reference precision of the library
        _case("2d-128-fp64", "prop", 128, 20, nt=150, y=1.3, prec="fp64"),
        # one product of the Newton-Krylov iteration: four illuminations on the 80^2 reconstruction grid
        _case("jvp-80-b4", "jvp", 80, 20, batch=4, nt=400, dx=0.125, ns=158),
        # an uneven grid whose FFT extents (150 x 210) have no specialised plan, without absorption
        _case("2d-uneven-lossless", "prop", "110,170", 20, batch=2, nt=200, lossless=True, ns=96),
        # a single 512^2 problem: one illumination, one direction
        _case("2d-512-b1", "prop", 512, 32, nt=250, dx=0.05, ns=256, sensors="perimeter"),
        # the production batch on that grid: twelve illuminations or Krylov directions at once
        _case("2d-512-b12", "prop", 512, 32, batch=12, nt=150, dx=0.05, ns=256, sensors="perimeter"),
        # differentiable use on the largest 2D grid, four illuminations: forward and backward
        _case("grad-1024-b4", "grad", 1024, 28, batch=4, nt=80, dx=0.05, ns=512, sensors="perimeter"),
        # Jacobian products on the three uneven grids of an inexact-Newton inner loop, 16 each
        _case("group-jvp-3x16", "group", "256,384,512", 16, batch=16, nt=80, dx=0.05, ns=256, sensors="perimeter"),
        # 3D: the 33^3-sized reconstruction grid with three illuminations
        _case("3d-32-b3", "prop", "3d:32", 8, batch=3, nt=150, dx=0.3, ns=400),
        # 3D at production size, the whole map: fluence solve and propagation on 256^3 (288^3 with the layer)
        _case("forward-3d-256", "forward", "3d:256", 16, nt=24, ns=4096, y=1.3),
        # the fluence solves of eight absorption maps on 512^2
        _case("da-512-b8", "da", 512, 32, batch=8, prec="fp64"),
        # the gradient in sound speed and density on the 128^2 grid, double precision
        _case("medium-128-fp64", "medium", 128, 20, nt=100, y=1.3, prec="fp64"),
    ]


def _smooth(n):
    for q in (2, 3, 5, 7):
        while n % q == 0:
            n //= q
    return n == 1


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _axis(rng, lo, hi, pml):
    """An even interior extent whose FFT extent factors into 2, 3, 5, 7 (half of them powers of two times 3)."""
    while True:
        n = _log_int(rng, lo, hi) // 2 * 2
        if n >= lo and _smooth(n + 2 * pml):
            return n


def draw(rng):
    kind = rng.choice(["prop", "prop", "prop", "prop", "prop3", "jvp", "grad", "da", "forward", "medium"])
    y = rng.choice([1.1, 1.3, 1.5])
    lossless = rng.random() < 0.2
    prec = "fp64" if rng.random() < 0.2 else "fp32"
    pml = rng.choice([8, 12, 16, 20, 24, 28, 32])
    if kind == "prop3":
        pml = rng.choice([4, 8, 12, 16])
        n = [_axis(rng, 12, 128, pml) for _ in range(3)] if rng.random() < 0.4 else [_axis(rng, 12, 128, pml)] * 3
        text, kind = "3d:" + ",".join(map(str, n)), "prop"
        batch = rng.choice([1, 1, 2, 3, 4])
    else:
        hi = {"da": 1024, "medium": 256, "jvp": 512, "forward": 512}.get(kind, 1024)
        hi = 256 if prec == "fp64" and kind != "da" else hi
        n0 = _axis(rng, 24, hi, pml)
        n = [n0, _axis(rng, max(24, n0 // 2), min(hi, 2 * n0), pml)] if rng.random() < 0.4 else [n0, n0]
        text = ",".join(map(str, n))
        batch = 1 if kind == "medium" else rng.choice([1, 1, 2, 3, 4, 6, 8, 12])
    if kind == "medium":
        prec = "fp64"           # the entry point returns double precision
    cells = batch
    for v in n:
        cells *= v + 2 * pml
    if kind == "da":
        nt = 2
        while batch > 1 and cells > 4e6:
            cells, batch = cells / batch, 1
    else:
        budget = 5e8 if prec == "fp32" else 6e6 if kind == "medium" else 5e7
        while batch > 1 and cells * 24 > budget:
            cells, batch = cells / batch, 1
        nt = int(max(8, min(400, budget / cells)))
    c = _case("", kind, text, pml, batch=batch, nt=nt, prec="fp64" if kind == "da" else prec, y=y, lossless=lossless,
              ns=rng.choice([33, 64, 128, 158, 256]), dx=rng.choice([0.05, 0.1, 0.125]))
    del c["name"]
    return c


# --------------------------------------------------------------------------------------------------
# inputs, made on the GPU from the seed

def _extents(text):
    """Interior shapes, x last: one tuple per grid ("a,b,c" of a group case is three square grids)."""
    if text.startswith("3d:"):
        v = [int(t) for t in text[3:].split(",")]
        return tuple(v * 3)[:3][::-1] if len(v) == 1 else tuple(v[::-1])
    v = [int(t) for t in text.split(",")]
    return (v[0], v[0]) if len(v) == 1 else tuple(v[::-1])


def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1000003 + salt)
    return g


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _coords(shape):
    """Node coordinates in units of dx, centred, one broadcastable tensor per axis, x first."""
    out = []
    for ax in range(len(shape) - 1, -1, -1):
        v = torch.arange(shape[ax], device=DEV, dtype=torch.float64) - (shape[ax] - 1) / 2.0
        out.append(v.view([-1 if a == ax else 1 for a in range(len(shape))]))
    return out


def _blobs(g, shape, extent, count, size):
    """`count` masks of axis-aligned ellipses inside the box `extent` (interior nodes, x first)."""
    co = _coords(shape)
    for _ in range(count):
        r2 = 0.0
        for ax, x in enumerate(co):
            centre = _uniform(g, -0.3, 0.3, 1).item() * extent[ax]
            semi = _uniform(g, *size, 1).item() * extent[ax]
            r2 = r2 + ((x - centre) / semi) ** 2
        yield r2 <= 1.0


def _problem(case, seed, interior, pml):
    """Medium, sensors and time step of one grid, FP64 on the GPU."""
    dim = len(interior)
    full = tuple(n + 2 * pml for n in interior)
    extent = interior[::-1]
    g = _gen(seed, 1)
    dx = case["dx"] * MM
    c = torch.full(full, 1500.0, dtype=torch.float64, device=DEV)
    rho = torch.full(full, 1000.0, dtype=torch.float64, device=DEV)
    alpha = torch.full(full, 0.75, dtype=torch.float64, device=DEV)
    for mask in _blobs(g, full, extent, 6, (0.04, 0.16)):
        c[mask] = _uniform(g, 1400.0, 1650.0, 1).item()
        rho[mask] = _uniform(g, 900.0, 1100.0, 1).item()
        alpha[mask] = _uniform(g, 0.5, 1.0, 1).item()
    kappa = torch.full(interior, MM / dim, dtype=torch.float64, device=DEV)
    for mask in _blobs(g, interior, extent, 2, (0.08, 0.2)):
        kappa[mask] = _uniform(g, 0.8, 1.2, 1).item() * MM / dim
    half = np.array([(n - 1) / 2.0 * dx for n in extent])
    ns = case["ns"]
    if case["sensors"] == "perimeter" and dim == 2:
        per = ns // 4
        t = -1.0 + 2.0 * np.arange(per) / per
        one = np.ones(per)
        pos = np.concatenate([np.stack(v, 1) for v in ((t, -one), (one, t), (-t, one), (-one, -t))]) * half
    elif dim == 2:
        th = 2 * np.pi * np.arange(ns) / ns
        pos = np.stack([np.cos(th), np.sin(th)], 1) * half * 0.85
    else:                        # a plane of detectors at the low-z face
        m = max(2, int(round(math.sqrt(ns))))
        t = np.linspace(-1.0, 1.0, m)
        Y, X = np.meshgrid(t, t, indexing="ij")
        pos = np.stack([X.ravel(), Y.ravel(), -np.ones(m * m)], 1) * half
    dt = 0.3 * dx / float(c.max())
    return dict(dim=dim, interior=interior, full=full, dx=dx, dt=dt, c=c, rho=rho, alpha=alpha, kappa=kappa, sensors=pos)


def _absorption(g, interior, batch):
    out = []
    for _ in range(batch):
        mu = torch.full(interior, 0.01 / MM, dtype=torch.float64, device=DEV)
        for mask in _blobs(g, interior, interior[::-1], 3, (0.05, 0.12)):
            mu[mask] = _uniform(g, 0.02, 0.05, 1).item() / MM
        out.append(mu)
    return torch.stack(out)


def _pressure(g, interior, batch, dtype):
    """An initial pressure: the heating of a tissue lit from its sides, strongest there, and a few Gaussian absorbers."""
    co = _coords(interior)
    out = []
    for _ in range(batch):
        p = torch.zeros(interior, dtype=torch.float64, device=DEV)
        for ax, x in enumerate(co):
            p += _uniform(g, 0.3, 0.7, 1).item() / len(co) * torch.cosh(6.0 * x / interior[::-1][ax]) / math.cosh(3.0)
        for _ in range(4):
            r2 = 0.0
            sig = _uniform(g, 0.03, 0.08, 1).item()
            for ax, x in enumerate(co):
                L = interior[::-1][ax]
                r2 = r2 + ((x - _uniform(g, -0.3, 0.3, 1).item() * L) / (sig * L)) ** 2
            p += _uniform(g, 0.5, 1.5, 1).item() * torch.exp(-r2 / 2.0)
        out.append(p)
    return torch.stack(out).to(dtype)


def _grids(case):
    if case["kind"] == "group":
        ns = [int(t) for t in case["n"].split(",")]
        return [((n, n), case["pml"] * n // ns[0]) for n in ns]
    return [(_extents(case["n"]), case["pml"])]


def _illum(dim):
    return (1 << (2 * dim)) - 1


def _inputs(case, seed):
    """Everything of a case that is not a handle of the library, per grid."""
    dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
    out = []
    for k, (interior, pml) in enumerate(_grids(case)):
        P = _problem(case, seed + 17 * k, interior, pml)
        g = _gen(seed, 100 + k)
        B, ns, kind = case["batch"], len(P["sensors"]), case["kind"]
        if kind in ("prop", "grad", "medium"):
            P["p0"] = _pressure(g, interior, B, dtype)
            # the series the adjoint is applied to: a residual, broad-band over sensors and time
            P["w"] = torch.randn(B, case["nt"], ns, generator=g, device=DEV, dtype=torch.float64).to(dtype)
        else:
            P["mu"] = _absorption(g, interior, B)
        if kind in ("jvp", "group"):
            P["dmu"] = torch.randn(B, *interior, generator=g, device=DEV, dtype=torch.float64) * 0.002 / MM
            # the fluence of the linearisation point, which a Newton iteration holds: here a smooth decay from the sides
            d = torch.ones(interior, dtype=torch.float64, device=DEV)
            for ax, x in enumerate(_coords(interior)):
                L = interior[::-1][ax]
                d = d * torch.cosh(2.0 * x / L) / math.cosh(1.0)
            P["phi0"] = (d * _uniform(g, 0.8, 1.2, B, *([1] * len(interior)))).contiguous()
        out.append(P)
    return out


# --------------------------------------------------------------------------------------------------
# one pass

def _context(case, P, pml):
    from paper_1810_11685_gb300 import binding
    host = [P[k].cpu().numpy() for k in ("c", "rho", "alpha", "kappa")]
    return binding.Context(host[0], host[1], None if case["lossless"] else host[2], host[3], P["sensors"], dx=P["dx"],
                           dt=P["dt"], nt=max(2, case["nt"]), pml=pml, y=case["y"], lossless=case["lossless"],
                           precision=case["prec"], max_batch=case["batch"])


def prepare(case, seed):
    from paper_1810_11685_gb300 import binding
    state = {"case": case, "in": _inputs(case, seed)}
    state["ctx"] = [_context(case, P, pml) for P, (_, pml) in zip(state["in"], _grids(case))]
    if case["kind"] == "group":
        state["group"] = binding.Group(state["ctx"])
    for P in state["in"]:        # the context holds the medium now
        for k in ("c", "rho", "alpha", "kappa"):
            del P[k]
    return state


def run(state):
    case, ctx, P = state["case"], state["ctx"][0], state["in"][0]
    kind = case["kind"]
    if kind == "prop":
        return {"data": ctx.acoustic_forward(P["p0"]), "p0_adj": ctx.acoustic_adjoint(P["w"])}
    if kind == "grad":
        from paper_1810_11685_gb300 import autograd
        p0 = P["p0"].detach().requires_grad_(True)
        data = autograd.acoustic(ctx, p0)
        (g,) = torch.autograd.grad(data, p0, P["w"])
        return {"data": data.detach(), "grad": g}
    if kind == "forward":
        return {"data": ctx.forward(P["mu"], _illum(P["dim"]))}
    if kind == "jvp":
        return {"dP": ctx.jvp(P["mu"], P["dmu"], _illum(P["dim"]), phi0=P["phi0"])}
    if kind == "group":
        ins = state["in"]
        outs = state["group"].jvp([Q["mu"] for Q in ins], [Q["dmu"] for Q in ins], _illum(2), [Q["phi0"] for Q in ins])
        return {"dP": outs}
    if kind == "da":
        return {"phi": ctx.da_solve(P["mu"], _illum(P["dim"]))}
    g_c, g_rho = ctx.vjp_medium(P["p0"], P["w"])
    return {"g_c": g_c, "g_rho": g_rho}


def work(case):
    """Inputs read once, outputs written once; flops: the real FFTs of every time step (2.5 N log2 N each)
    and the pointwise updates, and for a fluence solve the stencil of a handful of multigrid cycles."""
    elt = 8 if case["prec"] == "fp64" else 4
    B, nt, kind = case["batch"], case["nt"], case["kind"]
    nbytes = flops = 0.0
    for interior, pml in _grids(case):
        d = len(interior)
        N = float(np.prod(interior))
        G = float(np.prod([n + 2 * pml for n in interior]))
        ns = case["ns"]
        step_ffts = (1 + 2 * d + d) + (0 if case["lossless"] else 4)
        step = step_ffts * 2.5 * G * math.log2(G) + 20.0 * d * G
        medium = (2 + d + (0 if case["lossless"] else 2)) * G * elt
        series = B * nt * ns * elt
        da = 10 * 2 * (4 * d + 6) * N * B
        if kind in ("prop", "grad"):
            nbytes += 2 * (B * N * elt + series) + medium
            flops += 2 * B * nt * step
        elif kind == "medium":
            nbytes += N * 8 + series + 2 * G * 8 + medium
            flops += 2 * nt * step
        elif kind == "da":
            nbytes += 2 * B * N * 8 + (1 + d) * N * 8
            flops += da
        else:
            nbytes += (3 if kind != "forward" else 1) * B * N * 8 + series + medium + (1 + d) * N * 8
            flops += B * nt * step + da
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------------------------------
# the same in 64 bits with plain torch

def _wavenumbers(n, dx):
    m = torch.arange(n, device=DEV, dtype=torch.float64)
    return 2.0 * math.pi * torch.where(m < n / 2.0, m, m - n) / (n * dx)


def _pml(n, pml, dx, c_ref, dt, staggered):
    s = torch.arange(n, device=DEV, dtype=torch.float64) + (0.5 if staggered else 0.0)
    lo, hi = float(pml), float(n - pml - 1)
    xi = torch.clamp(lo - s, min=0.0) + torch.clamp(s - hi, min=0.0)
    return torch.exp(-2.0 * (c_ref / dx) * (xi / pml) ** 4 * dt / 2.0)


class _Exact:
    """The discretised acoustic map of one grid: forward loop and its transpose."""

    def __init__(self, case, P, pml):
        shape, dim, dx, dt = P["full"], P["dim"], P["dx"], P["dt"]
        self.shape, self.dim, self.dt, self.nt, self.lossless = shape, dim, dt, case["nt"], case["lossless"]
        c_ref = float(P["c"].max())
        y = case["y"]
        self.y = y
        self.alpha = P["alpha"] * 100.0 / (20.0 * math.log10(math.e)) / (2.0 * math.pi * 1e6) ** y
        view = lambda v, ax: v.view([-1 if a == ax else 1 for a in range(dim)])  # noqa: E731
        K = [view(_wavenumbers(shape[a], dx), a) for a in range(dim)]
        k = torch.sqrt(sum(q * q for q in K))
        x = c_ref * k * dt / 2.0
        kap = torch.where(x > 0, torch.sin(x) / torch.where(x > 0, x, torch.ones_like(x)), torch.ones_like(x))
        half = shape[-1] // 2 + 1
        self.Dp, self.Dm, self.An, self.As = [], [], [], []
        for i in range(dim):
            a = dim - 1 - i
            e = torch.exp(1j * K[a] * dx / 2.0)
            self.Dp.append((1j * K[a] * e * kap)[..., :half].contiguous())
            self.Dm.append((1j * K[a] * e.conj() * kap)[..., :half].contiguous())
            self.An.append(view(_pml(shape[a], pml, dx, c_ref, dt, False), a))
            self.As.append(view(_pml(shape[a], pml, dx, c_ref, dt, True), a))
        safe = torch.where(k > 0, k, torch.ones_like(k))
        self.Yd = torch.where(k > 0, safe ** (y - 1.0), torch.zeros_like(k))[..., :half].contiguous()
        self.Ya = torch.where(k > 0, safe ** (y - 2.0), torch.zeros_like(k))[..., :half].contiguous()
        self.inner = (Ellipsis,) + tuple(slice(pml, n - pml) for n in shape)
        self.set_medium(P["c"], P["rho"])
        # sensors: multilinear interpolation of the nodes
        pos = torch.from_numpy(np.ascontiguousarray(P["sensors"])).to(DEV)
        size = torch.tensor([shape[dim - 1 - i] for i in range(dim)], device=DEV)
        gpos = pos / dx + (size - 1) / 2.0
        base = torch.floor(gpos).long()
        frac = gpos - base
        idx, wgt = [], []
        for corner in range(1 << dim):
            flat, w, stride = 0, 1.0, 1
            for i in range(dim):
                b = (corner >> i) & 1
                flat = flat + torch.minimum(base[:, i] + b, size[i] - 1) * stride
                w = w * (frac[:, i] if b else 1.0 - frac[:, i])
                stride *= shape[dim - 1 - i]
            idx.append(flat)
            wgt.append(w)
        self.idx, self.wgt = torch.stack(idx), torch.stack(wgt)

    def set_medium(self, c, rho):
        self.C, self.rho0 = c * c, rho
        self.rs = [0.5 * (rho + torch.roll(rho, -1, dims=self.dim - 1 - i)) for i in range(self.dim)]
        if not self.lossless:
            self.tau = -2.0 * self.alpha * c ** (self.y - 1.0)
            self.eta = 2.0 * self.alpha * c ** self.y * math.tan(math.pi * self.y / 2.0)

    def fft(self, f):
        return torch.fft.rfftn(f, dim=tuple(range(-self.dim, 0)))

    def ifft(self, F):
        return torch.fft.irfftn(F, s=self.shape, dim=tuple(range(-self.dim, 0)))

    def sample(self, p):
        return (p.flatten(-self.dim)[..., self.idx] * self.wgt).sum(-2)

    def scatter(self, w):
        out = torch.zeros(w.shape[0], int(np.prod(self.shape)), dtype=torch.float64, device=DEV)
        for i, v in zip(self.idx, self.wgt):
            out.index_add_(1, i, w * v)
        return out.view(w.shape[0], *self.shape)

    def embed(self, p0):
        P0 = torch.zeros(*p0.shape[:-self.dim], *self.shape, dtype=torch.float64, device=DEV)
        P0[self.inner] = p0.double()
        return P0

    def forward(self, p0):
        """p0 [B][interior] -> [B][nt][ns]."""
        d, dt = self.dim, self.dt
        P0 = self.embed(p0)
        q = P0 / (2.0 * d * self.C)
        v = [torch.zeros_like(P0) for _ in range(d)]
        r = [torch.zeros_like(P0) for _ in range(d)]
        p = torch.zeros_like(P0)
        out = []
        for n in range(-1, self.nt - 1):
            F = self.fft(p)
            div = []
            for i in range(d):
                v[i] = self.As[i] * (self.As[i] * v[i] - dt / self.rs[i] * self.ifft(self.Dp[i] * F))
                div.append(self.ifft(self.Dm[i] * self.fft(v[i])))
                r[i] = self.An[i] * (self.An[i] * r[i] - dt * self.rho0 * div[i])
                if n <= 0:
                    r[i] = r[i] + q
            s = sum(r)
            if self.lossless:
                p = self.C * s
            else:
                u = sum(self.An[i] * self.rho0 * div[i] for i in range(d))
                p = self.C * (s - self.eta * self.ifft(self.Yd * self.fft(s)) + self.tau * self.ifft(self.Ya * self.fft(u)))
            out.append(self.sample(p))
        return torch.stack(out, 1)

    def adjoint(self, w):
        """w [B][nt][ns] -> [B][interior]: the transpose of forward."""
        d, dt = self.dim, self.dt
        w = w.double()
        zero = torch.zeros(w.shape[0], *self.shape, dtype=torch.float64, device=DEV)
        vb, rb = [zero.clone() for _ in range(d)], [zero.clone() for _ in range(d)]
        pb, qb = zero.clone(), zero.clone()
        for n in range(self.nt - 2, -2, -1):
            Cp = self.C * (pb + self.scatter(w[:, n + 1]))
            part, ub = Cp, None
            if not self.lossless:
                part = Cp - self.ifft(self.Yd * self.fft(self.eta * Cp))
                ub = self.ifft(self.Ya * self.fft(self.tau * Cp))
            F = 0
            for i in range(d):
                t = rb[i] + part
                g = -dt * self.rho0 * self.An[i] * t
                if ub is not None:
                    g = g + self.rho0 * self.An[i] * ub
                rb[i] = self.An[i] * self.An[i] * t
                if n <= 0:
                    qb += t
                vt = vb[i] + self.ifft(self.Dm[i].conj() * self.fft(g))
                vb[i] = self.As[i] * self.As[i] * vt
                F = F - self.Dp[i].conj() * self.fft(self.As[i] * dt / self.rs[i] * vt)
            pb = self.ifft(F)
        return (qb / (2.0 * d * self.C))[self.inner]


class _Fluence:
    """The finite-volume diffusion system of one grid, solved by conjugate gradients."""

    def __init__(self, P, mu):
        k, h, dim = P["kappa"], P["dx"], P["dim"]
        gam = 0.25 if dim == 3 else 1.0 / math.pi
        hf, hb, self.hd = h ** (dim - 2), h ** (dim - 1), h ** dim
        self.dim, diag = dim, torch.zeros_like(k)
        self.rhs0 = torch.zeros_like(k)
        self.face = []
        for a in range(dim):
            n = k.shape[a]
            lo, hi = k.narrow(a, 0, n - 1), k.narrow(a, 1, n - 1)
            f = 2.0 * lo * hi / (lo + hi) * hf
            diag.narrow(a, 0, n - 1).add_(f)
            diag.narrow(a, 1, n - 1).add_(f)
            self.face.append(f)
            for s in (0, n - 1):
                e = k.narrow(a, s, 1)
                diag.narrow(a, s, 1).add_(2.0 * gam * e * hb / (gam * h + e))
                self.rhs0.narrow(a, s, 1).add_(2.0 * e * hb / (gam * h + e))
        self.diag = diag + mu * self.hd

    def apply(self, x):
        y = self.diag * x
        for a, f in enumerate(self.face):
            ax = a - self.dim
            n = x.shape[ax]
            y.narrow(ax, 0, n - 1).sub_(f * x.narrow(ax, 1, n - 1))
            y.narrow(ax, 1, n - 1).sub_(f * x.narrow(ax, 0, n - 1))
        return y

    def solve(self, b):
        dims = tuple(range(-self.dim, 0))
        dot = lambda u, v: (u * v).sum(dims, keepdim=True)  # noqa: E731
        x, r = torch.zeros_like(b), b.clone()
        z = r / self.diag
        p, rz, bb = z.clone(), dot(r, z), dot(b, b)
        for it in range(20000):
            q = self.apply(p)
            al = rz / dot(p, q)
            x = x + al * p
            r = r - al * q
            z = r / self.diag
            new = dot(r, z)
            p = z + new / rz * p
            rz = new
            if it % 50 == 49 and bool((dot(r, r) <= 1e-29 * bb).all()):
                break
        return x


def exact(case, seed):
    outs = []
    for P, (_, pml) in zip(_inputs(case, seed), _grids(case)):
        kind = case["kind"]
        if kind == "da":
            S = _Fluence(P, P["mu"])
            return {"phi": S.solve(S.rhs0.expand_as(P["mu"]).clone())}
        E = _Exact(case, P, pml)
        if kind == "prop":
            return {"data": E.forward(P["p0"]), "p0_adj": E.adjoint(P["w"])}
        if kind == "grad":
            return {"data": E.forward(P["p0"]), "grad": E.adjoint(P["w"])}
        if kind == "medium":
            c, rho = P["c"].requires_grad_(True), P["rho"].requires_grad_(True)
            E.set_medium(c, rho)
            g = torch.autograd.grad(E.forward(P["p0"]), (c, rho), P["w"].double())
            return {"g_c": g[0], "g_rho": g[1]}
        S = _Fluence(P, P["mu"])
        if kind == "forward":
            return {"data": E.forward(P["mu"] * S.solve(S.rhs0.expand_as(P["mu"]).clone()))}
        dphi = S.solve(-S.hd * P["dmu"] * P["phi0"])
        outs.append(E.forward(P["dmu"] * P["phi0"] + P["mu"] * dphi))
    return {"dP": outs[0] if case["kind"] == "jvp" else outs}
