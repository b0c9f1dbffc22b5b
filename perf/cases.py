"""What a user of this package has it do, as measurable cases.

A case is one pass of a solidification run through the public entry points
(``native.Sim``, ``batch.Batch``): some time steps of one instance or of a
batch, returning psi and U of every instance, or the reductions of an observe.
Tiles are the library's own choice, as in the README's examples.

``exact`` evaluates the same steps in plain torch FP64 from the equations:
  a_s^2 F1 dpsi/dt = div J - sqrt2 phi a_s^2 |grad psi|^2 + sqrt2 [phi - lambda (1 - phi^2) F2]
  U' = U + [dt (D div[(1 - phi) grad U] + A) + (1 + (1-k) U) dphi] / (1 + k - (1-k) phi')
"""
import math

import numpy as np
import torch

from paper_2110_12448_gb300 import native, synth
from paper_2110_12448_gb300.batch import Batch

SQ2 = math.sqrt(2.0)
A1 = 5.0 * math.sqrt(2.0) / 8.0


def _case(name, what, **kw):
    c = {"what": what, "dim": 2, "nx": 0, "ny": 0, "nz": 1, "hi": 0, "count": 1, "scheme": "SBAR21", "precision": "f32",
         "steps": 1, "grains": 1, "phys": "dendrite", "directional": False, "time_level": 0, "sizes": 0}
    if name:
        c["name"] = name
    c.update(kw)
    return c


def listed():
    return [
        # the smallest runs a served stream holds (sides from 128): one small instance, two steps at a time,
        # where launches and latency count
        _case("single2d_128_f32", "step", nx=128, ny=128, steps=2),
        # the plain FP64 free dendrite that every precision is compared with
        _case("single2d_200_f64", "step", nx=200, ny=200, precision="f64", steps=4),
        # the README's first example: one 1024^2 instance
        _case("single2d_1024_f32", "step", nx=1024, ny=1024, steps=8),
        # the orientation sweep, the headline batch
        _case("sweep2d_10x1024_f32", "step", nx=1024, ny=1024, count=10, steps=16),
        # the same batch on the compensated state that meets the accuracy contract
        _case("sweep2d_10x1024_f32c", "step", nx=1024, ny=1024, count=10, steps=4, precision="f32c"),
        # the paper's isothermal 2D runs with the standard anti-trapping: an odd width, ten angles
        _case("paper2d_s21_10x781_f32", "step", nx=781, ny=781, count=10, steps=16, scheme="S21", phys="paper"),
        # polycrystals of ragged sizes, several grains each (the grain map is read)
        _case("poly2d_16_f32", "step", nx=256, ny=0, hi=1536, count=16, steps=16, grains=8, sizes=1),
        # directional solidification: frozen gradient, periodic x
        _case("directional2d_5x1024x2048_f32", "step", nx=1024, ny=2048, count=5, steps=16, directional=True),
        # the 3D free dendrite
        _case("dendrite3d_256_f32", "step", dim=3, nx=256, ny=256, nz=256, scheme="SBAR120", steps=4),
        # the anisotropic 3D scheme on a box of unequal, odd sides
        _case("dendrite3d_s100_157x121x189_f32", "step", dim=3, nx=157, ny=121, nz=189, scheme="S100", steps=4),
        # the 3D half of a served stream: polycrystals of ragged sides in one batch
        _case("poly3d_4_f32", "step", dim=3, nx=64, hi=192, count=4, scheme="SBAR120", steps=4, grains=6, sizes=2),
        # tip, growth angle, solute and solid fraction of every member of the sweep (a run observes every 100 steps)
        _case("observe2d_10x1024_f32", "observe", nx=1024, ny=1024, count=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sides over their logarithm, odd ones among them."""
    prec = rng.choice(["f32", "f32", "f32", "f32", "f64", "f32c"])
    if rng.random() < 0.3:
        lo, hi = (24, 72) if prec == "f64" else (32, 224)
        return _case(None, "step", dim=3, nx=_log(rng, lo, hi), ny=_log(rng, lo, hi), nz=_log(rng, lo, hi),
                     scheme=rng.choice(["SBAR120", "SBAR120", "S100"]), precision="f64" if prec == "f64" else "f32",
                     steps=rng.choice([1, 2, 4]), grains=rng.choice([1, 1, 5]), time_level=rng.choice([0, 0, 0, 1]))
    n, count = _log(rng, 96, 2048), rng.choice([1, 1, 2, 5, 10])
    most = 6e5 if prec == "f64" else 1e7
    m = _log(rng, max(64, n // 2), n * 2)
    while n * m * count > most:
        n, m = int(n * 0.7), int(m * 0.7)
    what = "observe" if rng.random() < 0.12 else "step"
    flavour = rng.random()
    grains, directional, level = 1, False, 0
    if flavour < 0.2:
        grains = rng.randint(3, 12)
    elif flavour < 0.4 and prec != "f32c":
        directional = True
    elif flavour < 0.5 and prec != "f32c":
        level = 1
    return _case(None, what, nx=n, ny=m, count=count, precision=prec, scheme=rng.choice(["SBAR21", "SBAR21", "S21", "S10"]),
                 steps=1 if what == "observe" else rng.choice([1, 4] if prec == "f32c" else [1, 4, 16]), grains=grains, directional=directional, time_level=level)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _sides(case):
    """(nx, ny, nz) of every instance; ragged batches draw them from the case's own number."""
    if not case["sizes"]:
        return [(case["nx"], case["ny"], case["nz"])] * case["count"]
    r = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["count"]):
        n = int(r.integers(case["nx"], case["hi"] + 1))
        out.append((n, n, n if case["dim"] == 3 else 1))
    return out


def _physics(case):
    p = dict(h=0.8, dt=0.02, k=0.15, eps4=0.02, lam=10.0, U0=-0.55)
    if case["phys"] == "paper":  # W/d0* = 16, Omega = 0.43
        lam = 16.0 * A1 * (1.0 - 0.9 * 0.43) / 0.1
        p = dict(h=1.2, k=0.1, eps4=0.014, lam=lam, U0=-0.43, dt=0.8 * 1.2**2 / (4 * 0.6267 * lam))
    p["D"] = 0.6267 * p["lam"]
    if case["dim"] == 3:
        p["dt"] = 0.9 * p["h"] ** 2 / (6 * p["D"])
    if case["directional"]:
        p["U0"] = -1.0
    return p


def _axes(n, h, dev):
    return [torch.arange(k, dtype=torch.float64, device=dev) * h for k in n]


def _instance(case, n, rng, i):
    """One instance as a growing crystal leaves it: psi (the signed distance to star-shaped grains, or to a
    perturbed front), U (the solute's diffusion profile ahead of it), grain map (None: one grain), rotations, seeds."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    p, dim = _physics(case), case["dim"]
    x = _axes(n, p["h"], dev)
    X = [x[0][None, :], x[1][:, None]] if dim == 2 else [x[0][None, None, :], x[1][None, :, None], x[2][:, None, None]]
    ext = [k * p["h"] for k in n[:dim]]
    if case["directional"]:
        yT, theta = ext[1] / 8.0, rng.uniform(0.0, 45.0)
        front = torch.full_like(x[0], yT)
        for m in range(1, 7):
            front = front + 0.4 * torch.sin(2 * math.pi * m * x[0] / ext[0] + rng.uniform(0, 2 * math.pi))
        eta = X[1] - front[None, :]
        U = torch.where(eta < 0, torch.zeros_like(eta), -1.0 + torch.exp(-0.1 * eta.clamp(min=0.0) / p["D"]))
        return -eta, U, None, synth.rot2d(theta).reshape(1, 9), np.array([[ext[0] / 2, -80.0, 0.0, p["h"]]])
    g = case["grains"]
    rots, seeds, psi, gmap = [], [], None, None
    for q in range(g):
        R = synth.rot2d(rng.uniform(0, 90) if g > 1 else 5.0 * (i % 10) + rng.uniform(-1, 1)) if dim == 2 else synth.random_rot3(rng)
        c = [e * (0.5 + rng.uniform(-0.02, 0.02) if g == 1 else rng.uniform(0.1, 0.9)) for e in ext]
        r0 = min(ext) * (rng.uniform(0.1, 0.3) if g == 1 else rng.uniform(0.04, 0.1))
        d = [X[a] - c[a] for a in range(dim)]
        rr = torch.sqrt(sum(t * t for t in d))
        cr = [sum(float(R[b, a]) * d[b] for b in range(dim)) / r0 for a in range(dim)]  # crystal frame, over r0
        rho4 = (rr / r0) ** 4
        s = r0 * (1.0 + 0.2 * (4.0 * sum(t**4 for t in cr) - 3.0 * rho4) / (1.0 + rho4)) - rr
        psi = s if psi is None else torch.maximum(psi, s)
        rots.append(R.reshape(9))
        seeds.append(c + [0.0] * (3 - dim) + [r0])
    if g > 1:
        best = None
        for q, s in enumerate(seeds):  # a cell belongs to the grain of its nearest seed sphere
            v = s[3] - torch.sqrt(sum((X[a] - s[a]) * (X[a] - s[a]) for a in range(dim)))
            if best is None:
                best, gmap = v, torch.zeros(v.shape, dtype=torch.int64, device=dev)
            else:
                gmap = torch.where(v > best, q, gmap)
                best = torch.maximum(best, v)
    U = p["U0"] * (1.0 - torch.exp(psi.clamp(max=0.0) / (0.1 * min(ext))))
    U = U + 0.01 * torch.sin(X[0] * rng.uniform(0.05, 0.2)) * torch.cos(X[1] * rng.uniform(0.05, 0.2))
    return psi, U, gmap, np.stack(rots), np.array(seeds)


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    return [_instance(case, n, rng, i) for i, n in enumerate(_sides(case))]


def _frozen(case, n):
    """(Vp, lT, yT) of the frozen temperature, where there is one."""
    return (0.1, max(500.0, 2.0 * n[1] * 0.8), n[1] * 0.8 / 8.0) if case["directional"] else (0.0, 1.0, 0.0)


class _State:
    """The handle that a user's program keeps, and the views of its fields it has taken so far."""

    def __init__(self, case):
        self.case, self.views, self.batch, self.sim = case, {}, None, None

    def fields(self, sim):
        psi, U, _ = sim.device_fields()
        out = []
        for p in (psi, U):
            v = self.views.get(p)
            if v is None:
                dt, size = (torch.float64, 8) if sim.p.precision == 1 else (torch.float32, 4)
                many = sim.n_cells * (2 if sim.p.precision == 2 else 1)
                at = p - sim.mem.data_ptr()
                v = sim.mem[at:at + many * size].view(dt)
                v = self.views[p] = v.view(sim.shape) if sim.p.precision != 2 else v.view(2, *sim.shape)
            out.append(v)
        if sim.p.precision == 2:  # hi + lo, as FP64
            out = [v[0].double() + v[1] for v in out]
        return out


def prepare(case, seed):
    p, ws = _physics(case), []
    for n, (psi, U, _, rots, seeds) in zip(_sides(case), _inputs(case, seed)):
        Vp, lT, yT = _frozen(case, n)
        w = synth.Workload(case["dim"], n[0], n[1], n[2], p["h"], p["dt"], p["k"], p["eps4"], p["lam"], p["D"], p["U0"],
                           case["scheme"], seeds, np.arange(len(seeds), dtype=np.int16), rots,
                           np.concatenate([seeds[:, :3]]), bc_x=int(case["directional"]), thermal=int(case["directional"]),
                           Vp=Vp, lT=lT, yT=yT, psi_init=psi.cpu().numpy(), U_init=U.cpu().numpy())
        w.time_level = case["time_level"]
        ws.append(w)
    s = _State(case)
    if case["count"] == 1:
        s.sim = native.Sim.from_workload(ws[0], case["precision"])
    else:
        s.batch = Batch(ws, case["precision"], n_streams=2)
    torch.cuda.synchronize()
    return s


def run(state):
    case, sim, batch = state.case, state.sim, state.batch
    if case["what"] == "observe":
        obs = [sim.observe(0)] if sim is not None else batch.observe(0)
        return {"solute": np.array([o["solute"] for o in obs]), "solid_fraction": np.array([o["solid_fraction"] for o in obs]),
                "tip": np.array([o["tip"] for o in obs]), "tip_index": np.array([o["tip_index"] for o in obs])}
    if sim is not None:
        sim.step(case["steps"])
        members = [sim]
    else:
        batch.step(case["steps"])
        members = batch.members
    got = [state.fields(m) for m in members]
    return {"psi": [f[0] for f in got], "U": [f[1] for f in got]}


def work(case):
    """Each field read once and written once per pass (a pass's steps in between could stay on the chip); the
    floating-point operations of the stencils, counted per cell and step with every face flux formed once."""
    cells = sum(a * b * c for a, b, c in _sides(case))
    size = 4 if case["precision"] == "f32" else 8
    if case["what"] == "observe":
        return {"bytes": 2.0 * cells * size, "flops": 4.0 * cells}
    flops = {"SBAR21": 220, "S21": 300, "S10": 170, "SBAR120": 480, "S100": 330}[case["scheme"]]
    return {"bytes": cells * (4.0 * size + (2 if case["grains"] > 1 else 0)), "flops": float(flops) * cells * case["steps"]}


# --------------------------------------------------------------------------
# the same passes in plain torch FP64
# --------------------------------------------------------------------------
def _pad(f, per, w):
    """Cell-centred mirror walls on every axis (-1 -> 0, -2 -> 1), or periodic x."""
    for ax in range(f.dim()):
        n = f.shape[ax]
        i = torch.arange(-w, n + w, device=f.device)
        if per and ax == f.dim() - 1:
            i = i % n
        else:
            i = torch.where(i < 0, -1 - i, i)
            i = torch.where(i >= n, 2 * n - 1 - i, i)
        f = f.index_select(ax, i)
    return f


def _shifts(f, shape, w):
    """at(dx, dy[, dz]): the padded field seen from every cell."""
    def at(*d):
        d = tuple(reversed(d))
        return f[tuple(slice(w + o, w + o + n) for o, n in zip(d, shape))]
    return at


def _unit(dim, a, s=1):
    e = [0] * dim
    e[a] = s
    return e


def _add(*v):
    return [sum(t) for t in zip(*v)]


def _frame(R, g):
    """crystal components of a lab gradient"""
    d = len(g)
    return [sum(R[b][a] * g[b] for b in range(d)) for a in range(d)]


def _aniso(R, g, eps, h2):
    """(components in the crystal frame, their s_p = n_p^2, a_s, guard)"""
    c = _frame(R, g)
    r2 = sum(t * t for t in c)
    low = r2 * h2 < 1e-20
    s = [t * t / torch.where(low, torch.ones_like(r2), r2) for t in c]
    a = 1.0 - 3.0 * eps + 4.0 * eps * sum(t * t for t in s)
    return c, s, a, low


def _flux_minus_grad(R, g, eps, h2, ax):
    """component ax of J - g, J = d(a_s^2 |g|^2 / 2) / dg"""
    d = len(g)
    c, s, a, low = _aniso(R, g, eps, h2)
    q = sum(t * t for t in s)
    j = [c[p] * (a * a - 1.0 - 16.0 * eps * a * q + 16.0 * eps * a * s[p]) for p in range(d)]
    out = sum(R[ax][p] * j[p] for p in range(d))
    return torch.where(low, torch.zeros_like(out), out)


def _face_gradient(at, ax, sg, h, dim):
    """two-point normal difference, four-point mean of centred differences across it, at the face toward sg along ax"""
    e, z, g = _unit(dim, ax, sg), [0] * dim, []
    for q in range(dim):
        if q == ax:
            g.append(sg * (at(*e) - at(*z)) / h)
        else:
            t, m = _unit(dim, q), _unit(dim, q, -1)
            g.append((at(*_add(e, t)) + at(*t) - at(*_add(e, m)) - at(*m)) / (4.0 * h))
    return g


def _div_shell(al, be, dim, h, iso, scale):
    """sum over the neighbours of (weighted alpha) (beta_e - beta_0) [scale(e): 1 / |grad| of the flux], over its h^2"""
    z, out = [0] * dim, 0.0
    edge = [[a, b] for a in (-1, 1) for b in (-1, 1)]
    for ax in range(dim):
        for sg in (-1, 1):
            e = _unit(dim, ax, sg)
            al_f = 0.5 * (al(*z) + al(*e))
            if iso and dim == 2:  # mean of the two corner means and the face mean, weight 4 in 6 h^2
                t = _unit(2, 1 - ax)
                m = [-v for v in t]
                K = [0.25 * (al(*z) + al(*e) + al(*o) + al(*_add(e, o))) for o in (t, m)]
                al_f = al(*z) + al(*e) + K[0] + K[1]
            elif iso:  # half the two-cell mean, the rest spread over the eight cells beside the pair, weight 2 in 6 h^2
                ring = 0.0
                for q in range(3):
                    if q != ax:
                        for s2 in (-1, 1):
                            t = _unit(3, q, s2)
                            ring = ring + al(*t) + al(*_add(e, t))
                al_f = 0.5 * (al(*z) + al(*e)) + 0.125 * ring
            f = al_f * (be(*e) - be(*z))
            out = out + (scale(e, f) if scale else f)
    if not iso:
        return out / (h * h)
    pairs = [(0, 1)] if dim == 2 else [(0, 1), (0, 2), (1, 2)]
    for a, b in pairs:
        for sa, sb in edge:
            ea, eb = _unit(dim, a, sa), _unit(dim, b, sb)
            e = _add(ea, eb)
            four = al(*z) + al(*ea) + al(*eb) + al(*e)
            if dim == 2:
                w = 0.25 * four
            else:
                c = 3 - a - b
                beside = 0.0
                for s2 in (-1, 1):
                    t = _unit(3, c, s2)
                    beside = beside + al(*t) + al(*_add(ea, t)) + al(*_add(eb, t)) + al(*_add(e, t))
                w = 3.0 / 16.0 * four + beside / 32.0
            f = w * (be(*e) - be(*z))
            out = out + (scale(e, f) if scale else f)
    return out / (6.0 * h * h)


def _grad_21(at, e, h):
    """the 21-point |grad psi| at the face or corner point e / 2 (coefficients of the standard anti-trapping scheme)"""
    if 0 in e:
        n, t = e, [abs(e[1]), abs(e[0])]

        def B(p, q):
            return at(*[p * n[i] + q * t[i] for i in range(2)])
        a1, a2 = B(1, 1) - B(0, -1), B(0, 1) - B(1, -1)
        b1, b2 = B(2, 1) - B(-1, -1), B(-1, 1) - B(2, -1)
        c1, c2 = B(1, 2) - B(0, -2), B(0, 2) - B(1, -2)
        u = (35.0 / 48.0 * (a1 - a2) - (b1 - b2) / 48.0 - (c1 - c2) / 6.0) / h
        v = (35.0 / 96.0 * (a1 + a2) - (b1 + b2) / 32.0 - (c1 + c2) / 24.0) / h
    else:
        def B(p, q):
            return at(p * e[0], q * e[1])
        a1, a2 = B(1, 1) - B(0, 0), B(0, 1) - B(1, 0)
        b1, b2 = B(2, 1) - B(-1, 0), B(-1, 1) - B(2, 0)
        c1, c2 = B(1, 2) - B(0, -1), B(0, 2) - B(1, -1)
        u = (0.625 * (a1 - a2) - (b1 - b2) / 48.0 - (c1 - c2) / 16.0) / h
        v = (0.625 * (a1 + a2) - (b1 + b2) / 16.0 - (c1 + c2) / 48.0) / h
    return torch.sqrt(u * u + v * v)


def _step(case, p, psi, U, R, zeta):
    dim, h, dt, k, eps, lam, D = case["dim"], p["h"], p["dt"], p["k"], p["eps4"], p["lam"], p["D"]
    scheme, per, h2, omk, shape = case["scheme"], case["directional"], h * h, 1.0 - k, psi.shape
    iso = scheme not in ("S10", "S100")
    P = _shifts(_pad(psi, per, 2), shape, 2)
    z = [0] * dim
    c = P(*z)
    faces = sum(P(*_unit(dim, a, s)) - c for a in range(dim) for s in (-1, 1))
    cen = [P(*_unit(dim, a)) - P(*_unit(dim, a, -1)) for a in range(dim)]
    g_face = sum(t * t for t in cen) / (4.0 * h2)
    if iso:
        pairs = [(0, 1)] if dim == 2 else [(0, 1), (0, 2), (1, 2)]
        diag = [_add(_unit(dim, a, sa), _unit(dim, b, sb)) for a, b in pairs for sa in (-1, 1) for sb in (-1, 1)]
        edges = sum(P(*e) - c for e in diag)
        g_edge = sum((P(*e) - P(*[-v for v in e])) ** 2 for e in diag) / 2.0
        if dim == 2:
            L, G = (4.0 * faces + edges) / (6.0 * h2), 2.0 / 3.0 * g_face + g_edge / (24.0 * h2)
        else:
            L, G = (2.0 * faces + edges) / (6.0 * h2), g_face / 3.0 + g_edge / (24.0 * h2)
    else:
        L, G = faces / h2, g_face
    N = 0.0
    for a in range(dim):
        for s in (-1, 1):
            N = N + s * _flux_minus_grad(R, _face_gradient(P, a, s, h, dim), eps, h2, a) / h
    _, _, a_s, low = _aniso(R, [t / (2.0 * h) for t in cen], eps, h2)
    a_s = torch.where(low, torch.ones_like(a_s), a_s)
    phi = torch.tanh(psi / SQ2)
    rate = (L + N + SQ2 * (phi - lam * (1.0 - phi * phi) * (U + zeta))) / (a_s * a_s) - SQ2 * phi * G
    rate = rate / (1.0 - omk * zeta)
    new = psi + dt * rate
    if case["time_level"]:
        dphi, phin = dt * (1.0 - phi * phi) / SQ2 * rate, phi
    else:
        phin = torch.tanh(new / SQ2)
        dphi = phin - phi
    aD = _shifts(_pad(1.0 - phi, per, 1), shape, 1)
    aA = _shifts(_pad((1.0 + omk * U) * dphi / (SQ2 * dt), per, 1), shape, 1)
    u = _shifts(_pad(U, per, 1), shape, 1)

    def over(m, f):
        low = m * m * h2 < 1e-20
        return torch.where(low, torch.zeros_like(f), f / torch.where(low, torch.ones_like(m), m))

    def standard(e, f):
        """a standard anti-trapping flux over |grad psi| at its point"""
        d = P(*e) - c
        if iso:
            ln = h * math.sqrt(sum(abs(v) for v in e))
            return over(torch.maximum(_grad_21(P, e, h), 0.5 * d.abs() / ln), f)
        ax = [i for i, v in enumerate(e) if v][0]
        g = _face_gradient(P, ax, e[ax], h, dim)
        return over(torch.sqrt(sum(t * t for t in g)), f)
    approx = scheme in ("SBAR21", "SBAR120")
    flux = D * _div_shell(aD, u, dim, h, iso, None) + _div_shell(aA, P, dim, h, iso, None if approx else standard)
    return new, U + (dt * flux + (1.0 + omk * U) * dphi) / (1.0 + k - omk * phin)


def _observed(psi, U, R, centre, p, dim):
    """solute integral, solid fraction and tip of the whole grid, axes of the one grain"""
    phi = torch.tanh(psi / SQ2)
    solute = float(((1 + p["k"] - (1 - p["k"]) * phi) * (1 + (1 - p["k"]) * U) / 2).sum()) * p["h"] ** dim
    axes = [[s * R[q][a] for q in range(dim)] for a in range(dim) for s in (1, -1)]
    d = max(axes, key=lambda v: v[1])
    ea = max(range(dim), key=lambda a: abs(d[a]))
    sg = 1 if d[ea] >= 0 else -1
    ax = dim - 1 - ea
    nxt = torch.roll(psi, -sg, ax)
    i = torch.arange(psi.shape[ax], device=psi.device).view([-1 if a == ax else 1 for a in range(dim)])
    ok = (psi >= 0) & (nxt < 0) & (i != (psi.shape[ax] - 1 if sg > 0 else 0))
    at = torch.nonzero(ok)
    pos = [at[:, dim - 1 - a].double() * p["h"] for a in range(dim)]
    ps, pn = psi[ok], nxt[ok]
    pos[ea] = pos[ea] + sg * ps / (ps - pn) * p["h"]
    score = sum((pos[a] - centre[a]) * d[a] for a in range(dim))
    b = int(score.argmax())
    return solute, float(((1 + phi) / 2).mean()), [float(t[b]) for t in pos] + [0.0] * (3 - dim)


def exact(case, seed):
    p, psis, us, seen = _physics(case), [], [], []
    for n, (psi, U, gmap, rots, seeds) in zip(_sides(case), _inputs(case, seed)):
        if case["precision"] == "f32":  # the state that the run starts from
            psi, U = psi.float().double(), U.float().double()
        dim = case["dim"]
        if case["what"] == "observe":
            if gmap is not None:
                return None
            R = rots[0].reshape(3, 3)
            seen.append(_observed(psi, U, R, seeds[0], p, dim))
            continue
        t = torch.tensor(rots, device=psi.device).view(-1, 3, 3)
        R = [[t[0, a, b] if gmap is None else t[:, a, b][gmap] for b in range(3)] for a in range(3)]
        Vp, lT, yT = _frozen(case, n)
        y = torch.arange(n[1], dtype=torch.float64, device=psi.device)[:, None] * p["h"]
        for s in range(case["steps"]):
            zeta = (y - yT - Vp * s * p["dt"]) / lT if case["directional"] else torch.zeros(1, dtype=psi.dtype, device=psi.device)
            psi, U = _step(case, p, psi, U, R, zeta)
        psis.append(psi)
        us.append(U)
    if case["what"] == "observe":
        return {"solute": np.array([o[0] for o in seen]), "solid_fraction": np.array([o[1] for o in seen]),
                "tip": np.array([o[2] for o in seen]), "tip_index": None}
    return {"psi": psis, "U": us}
