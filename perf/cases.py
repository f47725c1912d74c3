"""The work that a user of this library has it do, as cases that can be timed.

A case is one call, or one short sequence of calls, of the public binding
(paper_2101_05617_gb300.swepi) on one grid: the right-hand side, the
complex-step Jacobian-vector product in its full and its split form, the
phi-function solver, multistep EPI steps and the batched ensemble, in FP64 and
in the complex64-bulk form.  Grids and options are those of the repository's
workloads (6x4x4 p=3, 6x30x30 p=5, 6x60x60 p=5, 6x90x90 p=6, the ensemble's
n_e in {8, 16, 24, 32} x p in {3, 4, 5}) and sizes between them.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  a state: the context (grid tables, workspace) and the inputs on the GPU
  run(state)           one pass, and its outputs, one tensor per variable
  work(case)           bytes and floating-point operations one pass cannot do without
  exact(case, seed)    run's outputs from the plain FP64 restatement below

The restatement (Sphere, phi_sum, epi) is torch FP64 and shares nothing with
the library: panels are built from cube symmetry, interface fluxes are computed
on both sides of every interface in that side's own coordinates (the AUSM flux
of the other side is the same up to rounding), the product is a forward-mode
derivative and the phi-functions come from a fully orthogonalised Krylov space.
The inputs are made with it too, so they do not depend on the library's code.
"""
import math

import numpy as np
import torch

from paper_2101_05617_gb300 import swepi

RADIUS, GRAVITY, OMEGA = 6.37122e6, 9.80616, 7.292e-5
DEVICE = "cuda"
EPI_P = {3: 1, 4: 2, 5: 3, 6: 4}      # previous states an EPI order uses
EPI_M = {3: 2, 4: 3, 5: 4, 6: 4}      # phi-vectors phi_1 .. phi_M
EPI_A = {4: [[0.0, 0.0], [-3 / 10, 3 / 40], [32 / 5, -11 / 10]],
         5: [[0.0, 0.0, 0.0], [-4 / 5, 2 / 5, -4 / 45], [12.0, -9 / 2, 8 / 9], [3.0, 0.0, -1 / 3]],
         6: [[0.0, 0.0, 0.0, 0.0], [-49 / 60, 351 / 560, -359 / 1260, 367 / 6720],
             [92 / 7, -99 / 14, 176 / 63, -1 / 2], [485 / 21, -151 / 14, 23 / 9, -31 / 168]]}


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest grid of the repository: two launches, latency is all
        {"name": "rhs_ne4_p3", "kind": "rhs", "ne": 4, "p": 3, "topo": False},
        # the right-hand side every EPI step starts with, benchmark grid
        {"name": "rhs_ne60_p5", "kind": "rhs", "ne": 60, "p": 5, "topo": False},
        # the full complex-step product (one vector at a state), configuration 2's grid
        {"name": "jvp_ne30_p5", "kind": "jvp", "ne": 30, "p": 5, "topo": False},
        # an odd grid: a new linearisation point and the few products an EPI step's remainders take there
        {"name": "linearize_ne23_p4", "kind": "linearize", "ne": 23, "p": 4, "topo": True, "vectors": 3},
        # one split product at a held linearisation point: what every Krylov iteration is, benchmark grid and largest
        {"name": "product_ne60_p5", "kind": "product", "ne": 60, "p": 5, "topo": False, "form": "fp64"},
        {"name": "product_ne90_p6", "kind": "product", "ne": 90, "p": 6, "topo": True, "form": "fp64"},
        # the same in the complex64-bulk form
        {"name": "product_c64_ne60_p5", "kind": "product", "ne": 60, "p": 5, "topo": False, "form": "c64"},
        # a phi-function call of an EPI5 step on the benchmark grid, FP64 with the default window of two and the
        # complex64-bulk form with the window of three, the Krylov size warm from the call before (at 900 s: with
        # the benchmark's 1800 s the window-2 solver's step-size decisions turn on the last bit of its inputs)
        {"name": "phi_ne60_p5", "kind": "phi", "ne": 60, "p": 5, "form": "fp64", "iop": 2, "nb": 5, "dt": 900.0,
         "m": 128, "driver": 0},
        {"name": "phi_c64_ne60_p5", "kind": "phi", "ne": 60, "p": 5, "form": "c64", "iop": 3, "nb": 5, "dt": 900.0,
         "m": 128, "driver": 0},
        # whole EPI steps: the small configuration (host and launch latency) and configuration 2
        {"name": "epi4_ne4_p3", "kind": "epi", "ne": 4, "p": 3, "form": "fp64", "iop": 2, "order": 4, "dt": 900.0,
         "tol": 1e-12, "m": 16, "driver": 0},
        {"name": "epi5_ne30_p5", "kind": "epi", "ne": 30, "p": 5, "form": "fp64", "iop": 2, "order": 5, "dt": 1800.0,
         "tol": 1e-10, "m": 128, "driver": 0},
        # the batched ensemble, one member per class of the 96-member configuration
        {"name": "ensemble_12", "kind": "ensemble", "members": 12, "dt": 900.0, "m": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Grids from 4 to 80 elements a side and p = 2..6 (7 on small grids), every kind of call; steps as long as a
    Courant number of ten allows (the range in which the solver's step-size decisions are not decided by rounding)."""
    kind = rng.choice(["rhs", "jvp", "linearize", "product", "product", "phi", "phi", "epi", "epi"])
    p = rng.choice([2, 3, 3, 4, 5, 5, 6, 7])
    ne = _log_int(rng, 4, 80 if p <= 5 else 60)
    case = {"kind": kind, "ne": ne, "p": p}
    if kind in ("rhs", "jvp", "linearize", "product"):
        case["topo"] = rng.random() < 0.5
        if kind == "linearize":
            case["vectors"] = rng.randint(1, 4)
        if kind == "product":
            case["form"] = rng.choice(["fp64", "fp64", "c64"])
        return case
    case["ne"] = ne = min(ne, 48)
    spacing = RADIUS * math.pi / 2 / ne / (p + 1)
    case["dt"] = round(rng.uniform(2.0, 7.0) * spacing / 280.0, 1)
    case["form"] = "fp64" if kind == "epi" else rng.choice(["fp64", "fp64", "c64"])
    case["iop"] = 3 if case["form"] == "c64" else 2
    case["m"] = rng.choice([16, 32, 64, 96])
    case["driver"] = rng.choice([0, 0, 1])
    if kind == "phi":
        case["nb"] = rng.randint(2, 5)
    else:
        case["order"] = rng.choice([4, 5, 6])
        case["tol"] = rng.choice([1e-10, 1e-12])
    return case


# ------------------------------------------------------------------ inputs
def _grid_of(case, seed):
    rng = np.random.default_rng([seed, 1])
    rot = (rng.uniform(-math.pi, math.pi), rng.uniform(-math.pi / 3, math.pi / 3), rng.uniform(-math.pi, math.pi))
    return Sphere(case["ne"], case["p"], rot)


class Waves:
    """A smooth field on the sphere: plane waves of up to `degree` radians per radius, about `peak` at its largest."""

    def __init__(self, rng, degree, peak, count=12):
        d = rng.standard_normal((count, 3))
        d /= np.linalg.norm(d, axis=1, keepdims=True)
        self.k = torch.tensor(d * rng.uniform(1.0, degree, (count, 1)), device=DEVICE)
        self.ph = torch.tensor(rng.uniform(0, 2 * math.pi, count), device=DEVICE)
        self.a = torch.tensor(rng.standard_normal(count) * peak / (2.0 * math.sqrt(count)), device=DEVICE)

    def __call__(self, r):
        s = torch.zeros_like(r[0])
        for k, ph, a in zip(self.k, self.ph, self.a):
            s = s + a * torch.sin(k[0] * r[0] + k[1] * r[1] + k[2] * r[2] + ph)
        return s

    def grad(self, r):
        g = [torch.zeros_like(r[0]) for _ in range(3)]
        for k, ph, a in zip(self.k, self.ph, self.a):
            c = a * torch.cos(k[0] * r[0] + k[1] * r[1] + k[2] * r[2] + ph)
            g = [x + k[i] * c for i, x in enumerate(g)]
        return g


def _state(g, seed, topo):
    """A flow as it is some steps into an integration: 8000 m of fluid with a smooth anomaly, the wind geostrophic for
    it plus a divergent part of a few m/s, perhaps a bottom."""
    rng = np.random.default_rng([seed, 2])
    high = 4 if g.ne < 20 else 12
    anomaly, bottom, potential = Waves(rng, high, 150.0), Waves(rng, 8, 1000.0), Waves(rng, high, 2.0)
    r = g.r
    h = 8000.0 + anomaly(r)
    dh = anomaly.grad(r)
    f = GRAVITY / (2 * OMEGA * RADIUS)
    V = [f * (r[1] * dh[2] - r[2] * dh[1]), f * (r[2] * dh[0] - r[0] * dh[2]), f * (r[0] * dh[1] - r[1] * dh[0])]
    V = [a + b for a, b in zip(V, potential.grad(r))]
    hB = bottom(r) if topo else torch.zeros_like(h)
    c1, c2 = (sum(a * b for a, b in zip(V, t)) for t in (g.t1, g.t2))
    q0 = g.sg * (h - hB)
    return torch.stack([q0, q0 * (g.h11 * c1 + g.h12 * c2), q0 * (g.h12 * c1 + g.h22 * c2)]), hB


def _direction(g, q, seed, k):
    """What a Krylov space holds: smooth and rough parts together, each variable scaled like the state, 2-norm one."""
    rng = np.random.default_rng([seed, 3, k])
    gen = torch.Generator(device=DEVICE).manual_seed(int(rng.integers(1 << 60)))
    noise = torch.randn(q.shape, generator=gen, device=DEVICE, dtype=torch.float64)
    smooth = torch.stack([Waves(rng, 10, 2.0)(g.r) for _ in range(3)])
    v = (smooth + 0.2 * noise) * q.abs().mean(dim=(1, 2, 3, 4, 5), keepdim=True)
    return v / torch.linalg.vector_norm(v)


def _columns(g, q, seed, nb, dt):
    """b_0 .. b_{nb-1} of a phi-function call as an EPI step makes them: none, dt F, then small smooth remainders."""
    F = g.rhs(q)
    scale = F.abs().mean(dim=(1, 2, 3, 4, 5), keepdim=True)
    b = [None, dt * F]
    for k in range(2, nb):
        rng = np.random.default_rng([seed, 4, k])
        b.append(torch.stack([Waves(rng, 8, 0.05)(g.r) for _ in range(3)]) * scale * dt)
    return b[:nb]


def _history(g, q, order, dt):
    """(q_{n-i}, F(q_{n-i})) on the tangent through q_n: the previous states a multistep step reads."""
    F = g.rhs(q)
    qs = [q - i * dt * F for i in range(1, EPI_P[order] + 1)]
    return [(x, g.rhs(x)) for x in qs]


def _members(case, seed):
    out = []
    for k in range(case["members"]):
        out.append({"ne": (8, 16, 24, 32)[k % 4], "p": (3, 4, 5)[(k // 4) % 3], "order": 4 + (k + k // 4) % 2,
                    "seed": seed * 100 + k})
    return out


def _context(g, case, hB=None):
    ctx = swepi.SWContext(g.ne, g.p, g.rotation)
    if hB is not None and case.get("topo"):
        ctx.set_bottom(hB.reshape(-1).contiguous())
        g.set_bottom(hB)
    if case.get("form") == "c64":
        ctx.set_jvp_mode(2)
    if case.get("driver"):
        ctx.set_kiops_driver(1)
    return ctx


def _flat(x):
    return x.reshape(-1).contiguous()


def prepare(case, seed):
    if case["kind"] == "ensemble":
        ms = _members(case, seed)
        grids = [_grid_of(m, m["seed"]) for m in ms]
        qs = [_state(g, m["seed"], False)[0] for g, m in zip(grids, ms)]
        hist = [[(_flat(a), _flat(b)) for a, b in _history(g, q, m["order"], case["dt"])]
                for g, q, m in zip(grids, qs, ms)]
        ctxs = [_context(g, case) for g in grids]
        return {"case": case, "ens": swepi.SWEnsemble(ctxs), "ctxs": ctxs, "qs": [_flat(q) for q in qs], "hist": hist,
                "orders": [m["order"] for m in ms]}
    g = _grid_of(case, seed)
    q, hB = _state(g, seed, case.get("topo", False))
    ctx = _context(g, case, hB)
    s = {"case": case, "ctx": ctx, "q": _flat(q)}
    kind = case["kind"]
    if kind in ("jvp", "product"):
        s["v"] = _flat(_direction(g, q, seed, 0))
        s["out"] = torch.empty_like(s["v"])
        if kind == "product":
            ctx.linearize(s["q"])
    elif kind == "linearize":
        s["v"] = [_flat(_direction(g, q, seed, k)) for k in range(case["vectors"])]
        s["out"] = [torch.empty_like(x) for x in s["v"]]
    elif kind == "phi":
        s["b"] = [None if b is None else _flat(b) for b in _columns(g, q, seed, case["nb"], case["dt"])]
        s["out"] = torch.empty_like(s["q"])
    elif kind == "epi":
        s["hist"] = [(_flat(a), _flat(b)) for a, b in _history(g, q, case["order"], case["dt"])]
        s["y"] = torch.empty_like(s["q"])
    else:
        s["out"] = torch.empty_like(s["q"])
    return s


# ------------------------------------------------------------------ one pass
def _vars(x):
    """The mass and the two momentum densities."""
    return list(x.view(3, -1))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "rhs":
        return _vars(s["ctx"].rhs(s["q"], out=s["out"]))
    if kind == "jvp":
        return _vars(s["ctx"].jvp(s["q"], s["v"], out=s["out"]))
    if kind == "product":
        return _vars(s["ctx"].jvp_linearized(s["v"], out=s["out"]))
    if kind == "linearize":
        s["ctx"].linearize(s["q"])
        return [_vars(s["ctx"].jvp_linearized(v, out=o)) for v, o in zip(s["v"], s["out"])]
    if kind == "phi":
        w, _ = s["ctx"].kiops_phi(s["q"], case["dt"], s["b"], out=s["out"], tol=1e-10, m_init=case["m"],
                                  iop=case["iop"])
        return _vars(w)
    if kind == "epi":
        ctx = s["ctx"]
        ctx.epi_reset()
        for i, (a, b) in enumerate(s["hist"]):
            ctx.epi_set_history(i + 1, a, b)
        s["y"].copy_(s["q"])
        ctx.epi_step(case["order"], case["dt"], s["y"], tol=case["tol"], m_init=case["m"], iop=case["iop"])
        return _vars(s["y"])
    ys = []
    for ctx, q, hist in zip(s["ctxs"], s["qs"], s["hist"]):
        ctx.epi_reset()
        for i, (a, b) in enumerate(hist):
            ctx.epi_set_history(i + 1, a, b)
        ys.append(q.clone())
    s["ens"].epi_run(1, s["orders"], [case["dt"]] * len(ys), ys, m_init=case["m"])
    return [_vars(y) for y in ys]


# ------------------------------------------------------------------ what a pass cannot do without
def _product_work(nodes, ns, real=8):
    """A split product: v in, Jv out, the 11 node coefficients, 23 per interface point (12 N_s^2 / N_s per element
    and two sides each); per node the point fluxes and sources and 2 (N_s + 2) multiply-adds for three variables."""
    points = 2.0 * nodes / ns
    return {"bytes": nodes * (2 * 24 + 11 * real) + points * 23 * real,
            "flops": nodes * (26 + 12 * (ns + 2)) + points * (12 * ns + 40)}


def _nodes(case):
    return 6 * case["ne"] ** 2 * (case["p"] + 1) ** 2


def _iterations(case, ne, p, dt):
    """Krylov vectors a substep-free call needs at least: a few more than the Courant number of the grid's waves."""
    spacing = RADIUS * math.pi / 2 / ne / (p + 1)
    return max(10.0, 4.0 * 280.0 * dt / spacing)


def _phi_work(nodes, ns, nb, its, real=8):
    """Per Krylov vector a product that also reads the b columns, and the vector passes (V_j, V_{j-1} and z read, the
    new vector written; five multiply-adds per unknown); at the end the combination of the basis."""
    w = _product_work(nodes, ns, real)
    n = 3.0 * nodes
    return {"bytes": its * (w["bytes"] + n * ((nb - 1) * 8 + 24) + n * 8),
            "flops": its * (w["flops"] + n * (2 * (nb - 1) + 12))}


def _step_work(ne, p, order, dt):
    nodes, ns = 6 * ne ** 2 * (p + 1) ** 2, p + 1
    w = _phi_work(nodes, ns, EPI_M[order] + 1, _iterations(None, ne, p, dt))
    one = _product_work(nodes, ns)
    k = EPI_P[order] + 2
    return {"bytes": w["bytes"] + k * one["bytes"], "flops": w["flops"] + k * one["flops"]}


def work(case):
    if case["kind"] == "ensemble":
        parts = [_step_work(m["ne"], m["p"], m["order"], case["dt"]) for m in _members(case, 0)]
        return {k: sum(x[k] for x in parts) for k in ("bytes", "flops")}
    nodes, ns, kind = _nodes(case), case["p"] + 1, case["kind"]
    points = 2.0 * nodes / ns
    real = 4 if case.get("form") == "c64" else 8
    if kind == "rhs":     # q in, F out, 13 node and 12 interface coefficients
        return {"bytes": nodes * (48 + 104) + points * 96, "flops": nodes * (40 + 12 * (ns + 2)) + points * (12 * ns + 110)}
    if kind == "jvp":     # q and v in, Jv out; every real operation of the right-hand side with its imaginary half
        return {"bytes": nodes * (72 + 104) + points * 96, "flops": nodes * (110 + 12 * (ns + 2)) + points * (30 * ns + 180)}
    if kind == "product":
        return _product_work(nodes, ns, real)
    if kind == "linearize":
        w = _product_work(nodes, ns)
        return {"bytes": case["vectors"] * w["bytes"] + nodes * (24 + 104 + 88) + points * (96 + 144),
                "flops": case["vectors"] * w["flops"] + nodes * 40 + points * (12 * ns + 500)}
    if kind == "phi":
        return _phi_work(nodes, ns, case["nb"], _iterations(case, case["ne"], case["p"], case["dt"]), real)
    return _step_work(case["ne"], case["p"], case["order"], case["dt"])


# ------------------------------------------------------------------ the plain FP64 restatement
def _lagrange(nodes, x):
    """Values of the Lagrange basis of `nodes` at x."""
    return np.array([[np.prod([(xx - nodes[m]) / (nodes[k] - nodes[m]) for m in range(len(nodes)) if m != k])
                      for k in range(len(nodes))] for xx in x])


def _derivative(nodes, at):
    """d l_n / dx of the Lagrange basis of `nodes` at nodes[at]."""
    w = np.array([1.0 / np.prod([nodes[j] - nodes[k] for k in range(len(nodes)) if k != j])
                  for j in range(len(nodes))])
    D = np.zeros((len(nodes), len(nodes)))
    for i in range(len(nodes)):
        for j in range(len(nodes)):
            if i != j:
                D[i, j] = w[j] / w[i] / (nodes[i] - nodes[j])
        D[i, i] = -D[i].sum()
    return D[at]


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEVICE)


def _metric(X, Y, a=RADIUS):
    d2 = 1 + X * X + Y * Y
    return (a * a * (1 + X * X) * (1 + Y * Y) / d2 ** 1.5, d2 / (a * a * (1 + X * X)),
            X * Y * d2 / (a * a * (1 + X * X) * (1 + Y * Y)), d2 / (a * a * (1 + Y * Y)))


def _tangents(X, Y, frame, a=RADIUS):
    """Unit position and covariant basis vectors of the points (X, Y) of a panel, as lists of components."""
    c, e1, e2 = frame
    d = (1 + X * X + Y * Y) ** 0.5
    P = [c[k] + X * e1[k] + Y * e2[k] for k in range(3)]
    r = [x / d for x in P]
    t1 = [a * (1 + X * X) * (e1[k] / d - P[k] * X / d ** 3) for k in range(3)]
    t2 = [a * (1 + Y * Y) * (e2[k] / d - P[k] * Y / d ** 3) for k in range(3)]
    return r, t1, t2


class Sphere:
    """The rotated cubed sphere and the direct-flux-reconstruction right-hand side on it; arrays are
    [panel, e2, e1, k2, k1], states have the variable in front."""

    def __init__(self, ne, p, rotation):
        self.ne, self.p, self.ns, self.rotation = ne, p, p + 1, tuple(rotation)
        ns = p + 1
        lam, phi, al = rotation
        c = np.array([math.cos(phi) * math.cos(lam), math.cos(phi) * math.sin(lam), math.sin(phi)])
        el = np.array([-math.sin(lam), math.cos(lam), 0.0])
        ep = np.array([-math.sin(phi) * math.cos(lam), -math.sin(phi) * math.sin(lam), math.cos(phi)])
        a, b = math.cos(al) * el - math.sin(al) * ep, math.sin(al) * el + math.cos(al) * ep
        self.frames = [(c, a, b), (a, -c, b), (-c, -a, b), (-a, c, b), (b, a, -c), (-b, a, c)]
        xi, self.w = np.polynomial.legendre.leggauss(ns)
        ends = np.concatenate(([-1.0], xi, [1.0]))
        self.D = _dev(_derivative(ends, slice(1, ns + 1)))
        self.lm, self.lp = (_dev(v) for v in _lagrange(xi, (-1.0, 1.0)))
        self.Dg = _dev(_derivative(xi, slice(0, ns)))
        self.dx = math.pi / 2 / ne
        line = -math.pi / 4 + (np.arange(ne)[:, None] + 0.5 * (xi[None, :] + 1)) * self.dx
        t = np.tan(line)                                         # [ne, ns]
        faces = np.tan(-math.pi / 4 + np.arange(ne + 1) * self.dx)
        faces[0], faces[-1] = -1.0, 1.0
        shape = (6, ne, ne, ns, ns)
        X = _dev(t)[None, None, :, None, :].expand(shape)
        Y = _dev(t)[None, :, None, :, None].expand(shape)
        self.sg, self.h11, self.h12, self.h22 = (x.contiguous() for x in _metric(X, Y))
        fr = _dev(np.array(self.frames))                         # [panel, vector, component]
        fcol = [[fr[:, v, k].view(6, 1, 1, 1, 1) for k in range(3)] for v in range(3)]
        self.r, self.t1, self.t2 = _tangents(X, Y, fcol)
        d2 = 1 + X * X + Y * Y
        s = OMEGA / d2 * (fcol[0][2] + X * fcol[1][2] + Y * fcol[2][2])
        self.G0 = ((X * Y * s, -(1 + Y * Y) * s), ((1 + X * X) * s, -X * Y * s))
        self.Gs = ((2 * X * Y * Y / d2, -Y * (1 + Y * Y) / d2), (-X * (1 + X * X) / d2, 2 * X * X * Y / d2))
        # interface metric: x^1 = const faces [1, e2, ne + 1, k2] and x^2 = const faces [1, ne + 1, e1, k1]
        self.f1 = _metric(_dev(faces)[None, None, :, None], _dev(t)[None, :, None, :])
        self.f2 = _metric(_dev(t)[None, None, :, :], _dev(faces)[None, :, None, None])
        self.dB = None
        self._connect(t.reshape(-1))

    def _connect(self, t):
        """For each panel edge (W, E, S, N) the neighbouring panel's edge, its orientation and the transform of
        contravariant components from there."""
        one = np.ones_like(t)
        points = ((-one, t), (one, t), (t, -one), (t, one))
        self.near = {}
        for p in range(6):
            for e, (X, Y) in enumerate(points):
                r, t1, t2 = (np.array(v) for v in _tangents(X, Y, self.frames[p]))
                _, h11, h12, h22 = _metric(X, Y)
                dual = (h11 * t1 + h12 * t2, h12 * t1 + h22 * t2)
                mid = _tangents(np.array([X.mean()]), np.array([Y.mean()]), self.frames[p])[0]
                o = max((k for k in range(6) if k != p), key=lambda k: float(sum(mid[i][0] * self.frames[k][0][i] for i in range(3))))
                c, e1, e2 = self.frames[o]
                Xo, Yo = e1 @ r / (c @ r), e2 @ r / (c @ r)
                side = int(np.argmax([-Xo.mean(), Xo.mean(), -Yo.mean(), Yo.mean()]))
                along = Yo if side < 2 else Xo
                s1, s2 = (np.array(v) for v in _tangents(Xo, Yo, self.frames[o])[1:])
                T = [[(dual[i] * sj).sum(0) for sj in (s1, s2)] for i in range(2)]
                self.near[p, e] = (o, side, bool(along[0] > along[-1]), [[_dev(x) for x in row] for row in T])

    def set_bottom(self, hB):
        k = 2.0 / self.dx
        self.dB = (k * torch.einsum("kl,pefjl->pefjk", self.Dg, hB), k * torch.einsum("kl,pefli->pefki", self.Dg, hB))

    def _ghost(self, tr):
        """Traces of the neighbours at each panel edge, in this panel's components: [3][panel] of [ne, ns] per edge."""
        ne, ns = self.ne, self.ns
        edge = ((0, lambda a, o: a[o, :, 0]), (1, lambda a, o: a[o, :, -1]), (2, lambda a, o: a[o, 0]), (3, lambda a, o: a[o, -1]))
        out = []
        for e in range(4):
            per = [[], [], []]
            for p in range(6):
                o, side, back, T = self.near[p, e]
                q = [edge[side][1](tr[side][v], o).reshape(-1) for v in range(3)]
                if back:
                    q = [x.flip(0) for x in q]
                q = [q[0], T[0][0] * q[1] + T[0][1] * q[2], T[1][0] * q[1] + T[1][1] * q[2]]
                for v in range(3):
                    per[v].append(q[v].reshape(ne, ns))
            out.append([torch.stack(x) for x in per])
        return out

    @staticmethod
    def _ausm(L, R, d, m):
        sg, h11, h12, h22 = m
        hd = (h11, h12) if d == 1 else (h12, h22)
        hdd = hd[d - 1]

        def side(q):
            a = torch.sqrt(hdd * GRAVITY / sg * q[0])
            P = GRAVITY / (2 * sg) * q[0] * q[0]
            return a, q[d] / q[0] / a, (None, P * hd[0], P * hd[1])
        aL, ML, PL = side(L)
        aR, MR, PR = side(R)
        zero = torch.zeros_like(ML)
        inL, inR = ML.abs() <= 1, MR.abs() <= 1
        mp = torch.where(inL, 0.25 * (ML + 1) ** 2, torch.where(ML > 0, ML, zero))
        bp = torch.where(inL, 0.25 * (ML + 1) ** 2 * (2 - ML), torch.where(ML > 0, zero + 1, zero))
        mm = torch.where(inR, -0.25 * (MR - 1) ** 2, torch.where(MR > 0, zero, MR))
        bm = torch.where(inR, 0.25 * (MR - 1) ** 2 * (2 + MR), torch.where(MR > 0, zero, zero + 1))
        M = mp + mm
        out = []
        for k in range(3):
            adv = torch.where(M > 0, M * aL * L[k], M * aR * R[k])
            out.append(adv if k == 0 else adv + bp * PL[k] + bm * PR[k])
        return out

    def rhs(self, q):
        q0, q1, q2 = q[0], q[1], q[2]
        tr = [[torch.einsum("k,pefjk->pefj", l, x) for x in q] for l in (self.lm, self.lp)]
        tr += [[torch.einsum("k,pefkj->pefj", l, x) for x in q] for l in (self.lm, self.lp)]
        gh = self._ghost(tr)
        L = [torch.cat([gh[0][v][:, :, None], tr[1][v]], 2) for v in range(3)]
        R = [torch.cat([tr[0][v], gh[1][v][:, :, None]], 2) for v in range(3)]
        F1 = self._ausm(L, R, 1, self.f1)
        L = [torch.cat([gh[2][v][:, None], tr[3][v]], 1) for v in range(3)]
        R = [torch.cat([tr[2][v], gh[3][v][:, None]], 1) for v in range(3)]
        F2 = self._ausm(L, R, 2, self.f2)
        pre = GRAVITY / (2 * self.sg) * q0 * q0
        u1, u2 = q1 / q0, q2 / q0
        f12 = q1 * u2 + pre * self.h12
        flux = ((q1, q1 * u1 + pre * self.h11, f12), (q2, f12, q2 * u2 + pre * self.h22))
        G0, Gs = self.G0, self.Gs
        S = [None, -2 * (G0[0][0] * q1 + G0[0][1] * q2) - Gs[0][0] * q1 * u1 - 2 * Gs[0][1] * q1 * u2,
             -2 * (G0[1][0] * q1 + G0[1][1] * q2) - 2 * Gs[1][0] * q1 * u2 - Gs[1][1] * q2 * u2]
        if self.dB is not None:
            S[1] = S[1] - GRAVITY * q0 * (self.h11 * self.dB[0] + self.h12 * self.dB[1])
            S[2] = S[2] - GRAVITY * q0 * (self.h12 * self.dB[0] + self.h22 * self.dB[1])
        out = []
        for k in range(3):
            e1 = torch.cat([F1[k][:, :, :-1, :, None], flux[0][k], F1[k][:, :, 1:, :, None]], -1)
            e2 = torch.cat([F2[k][:, :-1, :, None, :], flux[1][k], F2[k][:, 1:, :, None, :]], -2)
            d = torch.einsum("kn,pefjn->pefjk", self.D, e1) + torch.einsum("kn,pefnj->pefkj", self.D, e2)
            out.append(-2.0 / self.dx * d if k == 0 else -2.0 / self.dx * d + S[k])
        return torch.stack(out)

    def jvp(self, q, v):
        return torch.func.jvp(self.rhs, (q,), (v,))[1]


def phi_sum(matvec, b, scale, m=80, tol=1e-14):
    """sum_k phi_k(A) b_k by the augmented exponential on [0, 1]: Krylov spaces of m fully orthogonalised vectors
    (twice), steps halved until the residual of the small exponential is below tol.  `scale` per variable makes the
    variables' sizes alike, so that the norm sees all of them."""
    shape = scale.shape
    full = next(x for x in b if x is not None)
    zero = torch.zeros_like(full)
    cols = [(zero if x is None else x) / scale for x in b]
    p, n = len(b) - 1, full.numel()
    mu = float(max(torch.linalg.vector_norm(x) for x in cols[1:])) or 1.0
    B = [x.reshape(-1) / mu for x in cols]
    assert shape[0] == 3

    def op(x):
        top = (matvec(x[:n].view_as(full) * scale) / scale).reshape(-1)
        for l in range(p):
            top = top + x[n + l] * B[p - l]
        return torch.cat([top, x[n + 1:], x.new_zeros(1)])

    x = torch.cat([cols[0].reshape(-1), full.new_zeros(p)])
    x[-1] = mu
    beta0 = float(torch.linalg.vector_norm(x))
    now = 0.0
    V = full.new_zeros((m + 1, n + p))
    while now < 1.0:
        beta = float(torch.linalg.vector_norm(x))
        V[0] = x / beta
        H = np.zeros((m + 1, m + 1))
        k = m
        for j in range(m):
            z = op(V[j])
            for _ in range(2):
                h = V[: j + 1] @ z
                z = z - h @ V[: j + 1]
                H[: j + 1, j] += h.cpu().numpy()
            H[j + 1, j] = float(torch.linalg.vector_norm(z))
            if H[j + 1, j] < 1e-13:
                k = j + 1
                break
            V[j + 1] = z / H[j + 1, j]
        tau = 1.0 - now
        while True:
            A = np.zeros((k + 1, k + 1))
            A[:k, :k] = H[:k, :k]
            A[0, k] = 1.0
            F = torch.linalg.matrix_exp(torch.tensor(tau * A))
            if k < m or beta * H[k, k - 1] * abs(float(F[k - 1, k])) <= tol * beta0 * tau or tau < 1e-6:
                break
            tau *= 0.7
        x = beta * (F[:k, 0].to(x.device) @ V[:k])
        now = 1.0 if now + tau > 1 - 1e-12 else now + tau
        for l in range(p):
            x[n + l] = mu * now ** (p - 1 - l) / math.factorial(p - 1 - l)
    return x[:n].view_as(full) * scale


def _scale(q):
    return q.abs().mean(dim=(1, 2, 3, 4, 5), keepdim=True)


def epi(g, q, hist, order, dt):
    """One multistep EPI step from q with the previous states `hist`."""
    F = g.rhs(q)
    R = [Fi - F - g.jvp(q, qi - q) for qi, Fi in hist]
    A = EPI_A[order]
    v = [sum(a * dt * r for a, r in zip(row, R)) for row in A]
    b = [None, dt * F + v[0]] + v[1:]
    return q + phi_sum(lambda x: dt * g.jvp(q, x), b, _scale(q))


def _three(x):
    return [y.reshape(-1) for y in x]


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        out = []
        for m in _members(case, seed):
            g = _grid_of(m, m["seed"])
            q, _ = _state(g, m["seed"], False)
            out.append(_three(epi(g, q, _history(g, q, m["order"], case["dt"]), m["order"], case["dt"])))
        return out
    g = _grid_of(case, seed)
    q, hB = _state(g, seed, case.get("topo", False))
    if kind in ("phi", "epi"):
        dt = case["dt"]
        if kind == "epi":
            return _three(epi(g, q, _history(g, q, case["order"], dt), case["order"], dt))
        return _three(phi_sum(lambda x: dt * g.jvp(q, x), _columns(g, q, seed, case["nb"], dt), _scale(q)))
    if case["topo"]:
        g.set_bottom(hB)
    if kind == "rhs":
        return _three(g.rhs(q))
    vs = [_direction(g, q, seed, k) for k in range(case["vectors"] if kind == "linearize" else 1)]
    out = [_three(g.jvp(q, v)) for v in vs]
    return out if kind == "linearize" else out[0]
