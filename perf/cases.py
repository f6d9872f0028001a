"""The work a user of the Vlasov--Poisson integrator has it do, as measurable cases.

A case is a plain dict: `kind` names the entry point (split steps, one adjoint
step, a whole trajectory gradient, the run's diagnostics), the sizes are the
six axis lengths, `dtype` the storage of f, `bc` the position boundary
("periodic", or "isolated": outflow faces and the doubled-grid Poisson solve),
`fixed` whether the time step is fixed, `steps` the split steps of one pass and
`kj` the ratio k/k_J of the longest mode (below 1 the box is Jeans unstable).

Ranges (`draw`): position axes of 4 to 64 cells, velocity axes of 6 to 64, or a
one-dimensional problem of up to 160 cells along x and vx with single cells
elsewhere; ragged and odd lengths as well as the powers of two and multiples of
16 that the configurations use; 2e4 to 1e9 cells in FP32, up to 1e8 in FP64.
Shifts stay below one cell per sweep, as the Courant limit makes them.
"""
import math

import numpy as np
import torch

from paper_1206_6152_gb300 import adjoint, vlasov

DEV = "cuda"
COURANT = 0.5
W0 = 6.0            # central potential of the isolated sphere, in sigma^2
TYPES = {"f32": torch.float32, "f64": torch.float64}


def _case(name, kind, n, nv, dtype="f32", bc="periodic", fixed=False, steps=1, kj=1.5):
    c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], vx=nv[0], vy=nv[1], vz=nv[2], dtype=dtype, bc=bc,
             fixed=fixed, steps=steps, kj=kj)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the 1D1V test problems run on degenerate six-dimensional grids:
        # many steps of a tiny state, all launches and latency
        _case("plane_wave_1d_f64", "step", (128, 1, 1), (128, 1, 1), "f64", steps=20),
        # gravitational Landau damping in FP64, the smallest 6D configuration
        _case("landau16_f64", "step", (16, 16, 16), (16, 16, 16), "f64", steps=4),
        # an odd small box in FP32, as someone tries a set-up out
        _case("ragged_small_f32", "step", (15, 12, 10), (18, 14, 13), steps=10),
        # an ordinary box whose lengths are none of the tuned ones
        _case("ragged_f32", "step", (20, 18, 22), (24, 28, 26), steps=2),
        # an ordinary production box: 32^3 velocity cells per spatial cell
        _case("jeans16x32_f32", "step", (16, 16, 16), (32, 32, 32), steps=5, kj=0.5),
        # the 32^6 Jeans box
        _case("jeans32_f32", "step", (32, 32, 32), (32, 32, 32), steps=4, kj=0.5),
        # a third of the 48^6 box of the benchmark, fixed step
        _case("jeans48_f32", "step", (16, 48, 48), (48, 48, 48), fixed=True, steps=2, kj=0.5),
        # fine velocity space: 64^3 velocity cells
        _case("velocity64_f32", "step", (16, 16, 16), (64, 64, 64), steps=2, kj=0.5),
        # isolated sphere with outflow faces, the merger's grid
        _case("isolated_f32", "step", (64, 32, 32), (32, 32, 32), bc="isolated", steps=2),
        # one adjoint step of the 32^6 fixed-step box (gradients of a long run)
        _case("adjoint32_f32", "adjoint", (32, 32, 32), (32, 32, 32), fixed=True, kj=0.5),
        # the whole gradient of a short trajectory through autograd
        _case("gradient16_f32", "gradient", (16, 16, 16), (32, 32, 32), fixed=True, steps=4, kj=0.5),
        # what a run prints at its output times: M, K, U, E and the density
        _case("diagnostics32_f32", "diagnostics", (32, 32, 32), (32, 32, 32), kj=0.5),
    ]


def _smooth(n):
    for p in (2, 3, 5, 7, 11, 13):
        while n % p == 0:
            n //= p
    return n == 1


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "step", "adjoint", "adjoint", "gradient",
                       "diagnostics"))
    if kind == "step" and rng.random() < 0.15:
        n = rng.choice([k for k in range(32, 161) if _smooth(k)])
        return _case(None, "step", (n, 1, 1), (rng.randint(32, 160), 1, 1), "f64",
                     steps=rng.randint(5, 20))
    dtype = "f64" if rng.random() < 0.25 else "f32"
    top = {"step": 5e8, "diagnostics": 1e9, "adjoint": 1.5e8, "gradient": 3e7}[kind]
    if dtype == "f64":
        top /= 10
    goal = math.exp(rng.uniform(math.log(2e4), math.log(top)))
    even = rng.random() < 0.5
    while True:
        if even:
            n = [rng.choice((16, 16, 32, 48, 8, 4)) for _ in range(3)]
            nv = [rng.choice((16, 32, 32, 48, 64))] * 3
        else:
            n = [int(math.exp(rng.uniform(math.log(4), math.log(65)))) for _ in range(3)]
            nv = [int(math.exp(rng.uniform(math.log(6), math.log(65)))) for _ in range(3)]
        cells = math.prod(n) * math.prod(nv)
        if 0.4 * goal <= cells <= 1.6 * goal and cells <= top and all(_smooth(k) for k in n):
            break
        even = even and rng.random() > 0.01     # small goals have no even grid
    bc = "isolated" if kind == "step" and rng.random() < 0.25 else "periodic"
    back = kind in ("adjoint", "gradient")
    steps = {"step": rng.randint(2, 4), "gradient": rng.randint(2, 5)}.get(kind, 1)
    return _case(None, kind, n, nv, dtype, bc, back or rng.random() < 0.3, steps,
                 rng.choice((0.5, 1.5)) if kind == "step" and cells > 1e8 else 1.5)


# ---------------------------------------------------------------------------
# geometry and inputs, from the case and the seed alone
# ---------------------------------------------------------------------------

class _Grid:
    def __init__(self, c):
        self.n = (c["nx"], c["ny"], c["nz"])
        self.nv = (c["vx"], c["vy"], c["vz"])
        self.isolated = c["bc"] == "isolated"
        big = max(self.n)
        self.rt = 17.0                              # radius of the isolated sphere
        length = 2.04 * self.rt if self.isolated else 1.0
        self.hi = tuple(0.5 * length * k / big for k in self.n)      # cubic cells
        self.lo = tuple(-h for h in self.hi)
        vb = 3.0 if self.isolated else 5.0
        self.vhi = tuple(vb if k > 1 else 0.5 for k in self.nv)
        self.vlo = tuple(-v for v in self.vhi)
        self.dx = tuple((h - l) / k for h, l, k in zip(self.hi, self.lo, self.n))
        self.dv = tuple((h - l) / k for h, l, k in zip(self.vhi, self.vlo, self.nv))
        self.G = 1.0
        kk = 2 * math.pi / length / c["kj"]
        self.rho_bar = kk * kk / (4 * math.pi * self.G)
        vmax = [max(abs(a), abs(b)) for a, b in zip(self.vlo, self.vhi)]
        self.dt_drift = min(h / v for h, v in zip(self.dx, vmax))
        self.dt_fixed = COURANT * self.dt_drift if c["fixed"] else 0.0

    def xc(self, a):
        return self.lo[a] + (np.arange(self.n[a]) + 0.5) * self.dx[a]

    def vc(self, a):
        return self.vlo[a] + (np.arange(self.nv[a]) + 0.5) * self.dv[a]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _outer3(a, b, c, op):
    return op(op(a[:, None, None], b[None, :, None]), c[None, None, :])


def _distribution(c, g, seed):
    """f at the cell centres: a Maxwellian with density modes and a small bulk
    velocity, or a lowered-isothermal sphere (zero beyond its escape speed)."""
    rng = np.random.default_rng(seed)
    u = rng.uniform(-0.2, 0.2, 3)
    v = [g.vc(a) - (u[a] if g.nv[a] > 1 else 0.0) for a in range(3)]
    f = torch.empty(g.n + g.nv, dtype=TYPES[c["dtype"]], device=DEV)
    flat = f.view(-1, math.prod(g.nv))
    step = max(1, (1 << 26) // flat.shape[1])
    if g.isolated:
        off = rng.uniform(-0.5, 0.5, 3)
        r = np.sqrt(_outer3(*[(g.xc(a) - off[a]) ** 2 for a in range(3)], np.add))
        psi = W0 * np.maximum((1 + r * r) ** -0.5 - (1 + g.rt ** 2) ** -0.5, 0.0)
        v2 = _outer3(*[t * t for t in v], np.add)
        norm = 9 / (4 * math.pi) / (np.maximum(np.expm1(W0 - v2 / 2), 0).sum() * math.prod(g.dv))
        psi, v2 = _dev(psi.reshape(-1)), _dev(v2.reshape(-1))
        for s in range(0, flat.shape[0], step):
            e = (psi[s:s + step, None] - 0.5 * v2[None, :]).clamp_(min=0.0)
            flat[s:s + step] = torch.expm1(e).mul_(norm)
        return f
    delta = np.zeros(g.n)
    for _ in range(3):
        k = [int(rng.choice((-2, -1, 1, 2))) if g.n[a] > 1 else 0 for a in range(3)]
        ph = _outer3(*[2 * math.pi * k[a] * g.xc(a) / (g.hi[a] - g.lo[a]) if g.n[a] > 1
                       else np.zeros(1) for a in range(3)], np.add)
        delta += rng.uniform(0.2, 1.0) * 1e-2 * np.cos(ph + rng.uniform(0, 2 * math.pi))
    m = [np.exp(-t * t / 2) / math.sqrt(2 * math.pi) if len(t) > 1 else np.ones(1) for t in v]
    rho, m = _dev(g.rho_bar * (1 + delta).reshape(-1)), _dev(_outer3(*m, np.multiply).reshape(-1))
    for s in range(0, flat.shape[0], step):
        flat[s:s + step] = rho[s:s + step, None] * m[None, :]
    return f


def _cotangents(c, g, seed):
    t = torch.Generator(device=DEV).manual_seed(seed + 1)
    lf = torch.randn(g.n + g.nv, dtype=TYPES[c["dtype"]], device=DEV, generator=t)
    lg = torch.randn((3,) + g.n, dtype=torch.float64, device=DEV, generator=t)
    return lf, lg


def prepare(case, seed):
    g = _Grid(case)
    f = _distribution(case, g, seed)
    cfg = vlasov.make_config(g.n, g.nv, g.lo, g.hi, g.vlo, g.vhi, G=g.G, courant=COURANT,
                             dt_fixed=g.dt_fixed, space_bc="outflow" if g.isolated else "periodic",
                             poisson_bc="isolated" if g.isolated else "periodic", dtype=f.dtype)
    s = dict(case=case, f0=f)
    if case["kind"] == "gradient":
        s["f0"] = f.requires_grad_(True)
        f = f.detach().clone()
    s["sim"] = vlasov.VlasovPoisson(cfg, f)
    if case["kind"] == "adjoint":
        s["g0"] = s["sim"].field()[2]
        s["lf"], s["lg"] = _cotangents(case, g, seed)
    return s


def run(state):
    kind, sim = state["case"]["kind"], state["sim"]
    if kind == "step":
        sim.step(state["case"]["steps"])
        return sim.f
    if kind == "adjoint":
        sim.adjoint_step(state["f0"], state["g0"], state["lf"], state["lg"])
        return {"lf": state["lf"], "lg": state["lg"]}
    if kind == "gradient":
        state["f0"].grad = None
        j = adjoint.trajectory_functional(state["f0"], sim, state["case"]["steps"], every=2)
        j.backward()
        return {"J": j.detach(), "grad": state["f0"].grad}
    e = sim.energy()
    return {"energy": {k: e[k] for k in ("M", "K", "U", "E")}, "rho": sim.density()}


def work(case):
    """A step needs the whole f of the step before it (through the field), so
    each step reads and writes f once; an adjoint step reads the step's f and
    reads and writes the cotangent.  Nine sweeps of about 15 operations a cell
    forward, about 40 more a sweep backward."""
    cells = math.prod(case[k] for k in ("nx", "ny", "nz", "vx", "vy", "vz"))
    size = cells * (4 if case["dtype"] == "f32" else 8)
    n = case["steps"]
    if case["kind"] == "step":
        return {"bytes": 2 * size * n, "flops": 136 * cells * n}
    if case["kind"] == "adjoint":
        return {"bytes": 3 * size, "flops": 9 * 55 * cells}
    if case["kind"] == "gradient":
        return {"bytes": 5 * size * n, "flops": (136 + 9 * 55) * cells * n}
    return {"bytes": size, "flops": 5 * cells}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the method's formulas
# ---------------------------------------------------------------------------

def _shift(f, d, by, periodic):
    """f displaced by one cell along d: entry i holds f[i - by]."""
    r = torch.roll(f, by, d)
    if not periodic:
        r.narrow(d, 0 if by > 0 else f.shape[d] - 1, 1).zero_()
    return r


def _update(f, alpha, d, periodic):
    """Positive-flux-conservative update of lines along d, |alpha| < 1."""
    b, neg = alpha.abs(), alpha < 0
    c1, c2 = b * (1 - b) * (2 - b) / 6, b * (1 - b) * (1 + b) / 6
    top = 2 * (f.amax(d, keepdim=True).clamp(min=0) - f)
    ep = torch.minimum(torch.maximum(_shift(f, d, -1, periodic) - f, -top), 2 * f)
    em = torch.minimum(torch.maximum(f - _shift(f, d, 1, periodic), -2 * f), top)
    phi = b * f + torch.where(neg, -c2, c1) * ep + torch.where(neg, -c1, c2) * em
    return f - phi + torch.where(neg, _shift(phi, d, -1, periodic), _shift(phi, d, 1, periodic))


class _Exact:
    def __init__(self, g):
        self.g = g
        self.per = not g.isolated
        n = g.n
        if g.isolated:
            self.m = tuple(2 * k if k > 1 else 1 for k in n)
            ax = [torch.minimum(torch.arange(m), m - torch.arange(m)).double().to(DEV) * h
                  for m, h in zip(self.m, g.dx)]
            r = _outer3(*[t * t for t in ax], torch.add).sqrt_()
            ker = -g.G / r
            ker[0, 0, 0] = -g.G * (3 * math.log(2 + math.sqrt(3)) - math.pi / 2) / g.dx[0]
            self.hat = torch.fft.fftn(ker).real * math.prod(g.dx)
        else:
            self.m = n
            s = [torch.sin(math.pi * torch.arange(m, dtype=torch.float64, device=DEV) / m) ** 2 / h ** 2
                 for m, h in zip(n, g.dx)]
            den = _outer3(*s, torch.add)
            den[0, 0, 0] = 1
            self.hat = -math.pi * g.G / den
            self.hat[0, 0, 0] = 0

    def density(self, f):
        rho = torch.empty(self.g.n, dtype=torch.float64, device=DEV)
        for i in range(self.g.n[0]):
            rho[i] = f[i].double().sum((2, 3, 4))
        return rho * math.prod(self.g.dv)

    def potential(self, rho):
        return torch.fft.ifftn(torch.fft.fftn(rho, self.m, dim=(0, 1, 2)) * self.hat).real

    def accel(self, rho):
        n, phi = self.g.n, self.potential(rho)
        a = [(torch.roll(phi, 1, k) - torch.roll(phi, -1, k)) / (2 * self.g.dx[k]) for k in range(3)]
        return torch.stack([t[:n[0], :n[1], :n[2]] for t in a])

    def dt(self, acc):
        if self.g.dt_fixed > 0:
            return self.g.dt_fixed
        m = max(float(acc[a].abs().max()) / self.g.dv[a] for a in range(3))
        return COURANT * min(self.g.dt_drift, 1 / m if m > 0 else math.inf)

    def alpha(self, axis, tau, acc):
        if axis < 3:
            shape = [1] * 6
            shape[3 + axis] = -1
            return (_dev(self.g.vc(axis)) * tau / self.g.dx[axis]).view(shape)
        return (acc[axis - 3] * tau / self.g.dv[axis - 3])[..., None, None, None]

    def pieces(self, f, axis):
        """(dimension, start, length) of the parts of f that one sweep takes at a time."""
        d = 3 if axis == 0 else 0
        per = f.numel() // f.shape[d]
        k = max(1, (1 << 27) // per)
        return [(d, s, min(k, f.shape[d] - s)) for s in range(0, f.shape[d], k)]

    @staticmethod
    def part(t, d, s, k):
        return t.narrow(d, s, k) if t.shape[d] > 1 else t

    def sweep(self, f, axis, tau, acc):
        a = self.alpha(axis, tau, acc)
        for p in self.pieces(f, axis):
            q = f.narrow(*p)
            q.copy_(_update(q, self.part(a, *p), axis, axis < 3 and self.per))

    def back(self, f, lam, axis, tau, acc):
        """lam: cotangent of the sweep's output, turned into its input's; returns that of acc."""
        a = self.alpha(axis, tau, acc)
        la = torch.zeros_like(a)
        for p in self.pieces(f, axis):
            x = f.narrow(*p).clone().requires_grad_(True)
            b = self.part(a, *p).clone().requires_grad_(axis >= 3)
            want = [x, b] if axis >= 3 else [x]
            got = torch.autograd.grad(_update(x, b, axis, axis < 3 and self.per), want, lam.narrow(*p))
            lam.narrow(*p).copy_(got[0])
            if axis >= 3:
                self.part(la, *p).add_(got[1])
        return la.reshape(self.g.n) * (tau / self.g.dv[axis - 3]) if axis >= 3 else None

    ORDER = ((3, 0.5), (4, 0.5), (5, 0.5), (2, 1.0), (1, 1.0), (0, 1.0), (3, 0.5), (4, 0.5), (5, 0.5))

    def step(self, f, acc, keep=None):
        dt = self.dt(acc)
        for k, (axis, part) in enumerate(self.ORDER):
            if k == 6:
                acc = self.accel(self.density(f))
            if keep is not None:
                keep.append(f.clone())
            self.sweep(f, axis, part * dt, acc)
        return acc

    def field_back(self, lg, lam):
        rho = torch.zeros(self.g.n, dtype=torch.float64, device=DEV, requires_grad=True)
        lr, = torch.autograd.grad(self.accel(rho), rho, lg)
        lam += (lr * math.prod(self.g.dv))[..., None, None, None]

    def step_back(self, f, acc, lam, lg):
        """(lam, lg): cotangents after the step, turned into those before it; f is used up."""
        kept, dt = [], self.dt(acc)
        after = self.step(f, acc, kept)
        for k in reversed(range(9)):
            axis, part = self.ORDER[k]
            la = self.back(kept.pop(), lam, axis, part * dt, after if k > 5 else acc)
            if la is not None:
                lg[axis - 3] += la
            if k == 6:
                self.field_back(lg, lam)
                lg.zero_()


def exact(case, seed):
    g = _Grid(case)
    f = _distribution(case, g, seed).double()
    x = _Exact(g)
    if case["kind"] == "diagnostics":
        rho = x.density(f)
        v2 = _dev(_outer3(*[g.vc(a) ** 2 for a in range(3)], np.add).reshape(-1))
        w = math.prod(g.dx) * math.prod(g.dv)
        m = float(rho.sum()) * math.prod(g.dx)
        k = sum(float((p @ v2).sum()) for p in f.view(g.n[0], -1, v2.numel())) * 0.5 * w
        n = g.n
        u = 0.5 * float((rho * x.potential(rho)[:n[0], :n[1], :n[2]]).sum()) * math.prod(g.dx)
        return {"energy": {"M": m, "K": k, "U": u, "E": k + u}, "rho": rho}
    acc = x.accel(x.density(f))
    if case["kind"] == "step":
        for _ in range(case["steps"]):
            acc = x.step(f, acc)
        return f
    if case["kind"] == "adjoint":
        lf, lg = _cotangents(case, g, seed)
        lf = lf.double()
        x.step_back(f, acc, lf, lg)
        return {"lf": lf, "lg": lg}
    start = []
    for _ in range(case["steps"]):
        start.append((f.clone(), acc))
        acc = x.step(f, acc)
    rho = x.density(f)
    n, phi = g.n, x.potential(rho)
    phi = phi[:n[0], :n[1], :n[2]]
    j = 0.5 * (rho * phi).sum() * math.prod(g.dx)
    lam = (phi * math.prod(g.dx) * math.prod(g.dv))[..., None, None, None].expand(f.shape).contiguous()
    lg = torch.zeros((3,) + g.n, dtype=torch.float64, device=DEV)
    del f
    while start:
        x.step_back(*start.pop(), lam, lg)
    x.field_back(lg, lam)
    return {"J": j, "grad": lam}
