"""The work that users of this framework have it do, as cases whose speed can be measured.

A case is a dict of plain values. Four kinds:

  pic      a particle-in-cell run: `steps` full steps of Sim.step (or one Sim.step_host, or steps
           with Sim.inject after each) on a seeded e+- plasma in a Wald or monopole field
  vacuum   the field solver alone (a run whose species hold no particles)
  push     test particles or photons through frozen fields, Sim.push without a deposit
  adjoint  gradients of test-particle orbits, push_adjoint forward and backward

Inputs (particles, perturbations, cotangents) are drawn on the GPU from the seed alone.
exact() computes the same results with plain torch in 64 bits, from the method's equations.

FP64 runs return the whole particle state and the field planes. In a mixed run the sums of FP32
currents have no fixed order, so a particle on a cell edge may be sorted into either cell, and
every particle behind it in the array moves: a mixed run that sorts returns the planes of the
fields and currents, one that does not (and the mixed test particles) the particles too, their
positions as one number each.
"""
from __future__ import annotations

import math

import torch
import torch.utils.checkpoint

import paper_2511_17701_gb300 as P

DEV = "cuda:0"
F8 = torch.float64
G = 2                       # ghost cells per side of a plane
LAST_J = (15, 16, 17)       # GRPIC_J01 .. GRPIC_J03
KEYS = ("i1", "i2", "dx1", "dx2", "u1", "u2", "u3", "phi", "w", "tag")
FIELDS = {"wald": P.FIELD_WALD, "monopole": P.FIELD_MONOPOLE}
R_H = 1.0 + math.sqrt(1.0 - 0.9 ** 2)   # horizon of the a = 0.9 runs

_PIC = dict(kind="pic", prec="fp64", a=0.9, n_r=512, n_theta=512, r_min=0.95 * R_H, r_max=50.0, ppc=32,
            theta=1.0, power=0.0, field="wald", rho0=1.0, d0=1.0, n_filter=0, sort_every=10,
            iter_tol=1e-12, r0=0.0, h0=0.0, steps=1, host=False, inject=False)
_BZ = dict(a=0.2, r_min=1.0, r_max=10.0, theta=0.5, power=2.0, field="monopole", rho0=5e-5, d0=2.5e-3)
SIGMA0, SIGMA_TH = 2500.0, 2000.0
POOL_N = 65536


def listed():
    return [
        # the smallest run, a first try or a test: 64^2 cells, filtered currents, ten steps and a sort
        dict(_PIC, name="pic_64_filter_fp64", n_r=64, n_theta=64, r_min=0.7 * R_H, r_max=10.0, ppc=8,
             theta=0.3, n_filter=4, steps=10),
        # the same size in mixed precision with the default options (no sort, no filter)
        dict(_PIC, name="pic_64_mixed", prec="mixed", n_r=64, n_theta=64, r_max=10.0, ppc=8, theta=0.1,
             sort_every=0, iter_tol=0.0, steps=10),
        # an ordinary run on a 512^2 grid, 16.8 M particles
        dict(_PIC, name="pic_512_fp64"),
        dict(_PIC, name="pic_512_mixed", prec="mixed", iter_tol=0.0, steps=10),
        # the largest: the benchmark's 2048^2 workload, 134 M particles
        dict(_PIC, name="pic_2048_fp64", n_r=2048, n_theta=2048, r_max=200.0, ppc=16, power=1.0),
        dict(_PIC, name="pic_2048_mixed", prec="mixed", n_r=2048, n_theta=2048, r_max=200.0, ppc=16,
             power=1.0, iter_tol=0.0, steps=10),
        # the monopole problem: strongly magnetised plasma, pair injection after the step
        {**_PIC, **_BZ, "name": "bz_512_fp64", "ppc": 8, "inject": True},
        # a run whose particles live in host memory and stream through the GPU each step
        dict(_PIC, name="host_512_fp64", ppc=8, host=True),
        # the field solver alone, as in vacuum tests and at start-up: a large grid, a small ragged one
        dict(kind="vacuum", name="vacuum_2048_fp64", prec="fp64", a=0.9, n_r=2048, n_theta=2048,
             r_min=0.95 * R_H, r_max=200.0, field="wald", r0=0.0, h0=0.0, n_filter=0, steps=10),
        dict(kind="vacuum", name="vacuum_500x300_mixed", prec="mixed", a=0.9, n_r=500, n_theta=300,
             r_min=0.95 * R_H, r_max=50.0, field="wald", r0=0.0, h0=0.0, n_filter=0, steps=10),
        # ray tracing: photons on a grid refined towards the equator, default options
        dict(kind="push", name="photons_qks_fp64", prec="fp64", a=0.9, n_r=512, n_theta=512,
             r_min=0.95 * R_H, r_max=50.0, field="wald", r0=0.4, h0=0.45, n=1000003, massless=True,
             iter_tol=0.0, theta=1.0, steps=4),
        # gradients of orbits with respect to their start and the field amplitude
        dict(kind="adjoint", name="adjoint_512", a=0.9, n_r=512, n_theta=512, r_min=0.95 * R_H, r_max=50.0,
             field="wald", n=65536, steps=100, every=25),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _r_min(a, n_r, r_max, r0, n_f):
    """An inner radius that puts the layer of n_f + 1 cells next to it inside the horizon."""
    r_h, q = 1.0 + math.sqrt(1.0 - a * a), (n_f + 1.5) / n_r
    return math.floor(1e4 * min(0.95 * r_h, r0 + (r_h - r0) ** (1 / (1 - q)) / (r_max - r0) ** (q / (1 - q)))) / 1e4


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["pic", "pic", "pic", "pic", "vacuum", "push", "adjoint"])
    a = round(rng.uniform(0.1, 0.97), 3)
    n_r, n_th = _log(rng, 48, 1100), _log(rng, 48, 1100)
    r_max = round(math.exp(rng.uniform(math.log(8.0), math.log(200.0))), 2)
    qks = dict(r0=round(rng.uniform(0.1, 0.5), 3), h0=round(rng.uniform(-0.2, 0.6), 3)) \
        if rng.random() < 0.25 else dict(r0=0.0, h0=0.0)
    if kind == "adjoint":
        n_r, n_th, qks = max(n_r, 200), max(n_th, 200), dict(r0=0.0, h0=0.0)
    grid = dict(a=a, n_r=n_r, n_theta=n_th, r_min=_r_min(a, n_r, r_max, qks["r0"], 0), r_max=r_max)
    prec = rng.choice(["fp64", "mixed"])
    field = rng.choice(["wald", "wald", "monopole"])
    if kind == "vacuum":  # a monopole's own B^2 and D are rounding only: in FP64 they stay far below the wave
        return dict(kind=kind, prec=prec, **grid, field=field if prec == "fp64" else "wald", **qks, n_filter=0, steps=rng.randint(1, 10))
    if kind == "push":
        return dict(kind=kind, prec=prec, **grid, field=field, **qks, n=_log(rng, 1000, 4000000),
                    massless=rng.random() < 0.5, iter_tol=rng.choice([0.0, 1e-12]),
                    theta=round(rng.uniform(0.1, 1.0), 2), steps=rng.randint(1, 4))
    if kind == "adjoint":
        n = _log(rng, 1000, 100000)
        return dict(kind=kind, **grid, field=field, n=n,
                    steps=rng.randint(8, 50), every=rng.randint(4, 30))
    c = _PIC | grid | qks | dict(prec=prec, field="wald", theta=round(rng.uniform(0.1, 1.0), 2),
                                              power=float(rng.randint(0, 2)))
    c["ppc"] = max(1, min(rng.randint(1, 40), 12000000 // (n_r * n_th)))
    form = rng.choice(["plain", "plain", "plain", "host", "bz", "filter"])
    if form == "host" or (form == "bz" and prec == "mixed"):
        c |= dict(prec="fp64")
    if form == "bz":
        c |= {**_BZ, "inject": True, "r0": 0.0, "h0": 0.0, "ppc": min(c["ppc"], 8), "r_min": _r_min(0.2, n_r, 10.0, 0.0, 0)}
    if form == "filter":
        n_f = rng.randint(1, 6)
        c |= dict(n_filter=n_f, r_min=_r_min(a, n_r, r_max, qks["r0"], n_f))
    c["host"] = form == "host"
    small = n_r * n_th * c["ppc"] < 1000000
    c["steps"] = rng.choice([1, 3, 10]) if small or prec == "mixed" else 1
    c["steps"] = 1 if c["host"] or c["inject"] else c["steps"]
    c["iter_tol"] = rng.choice([0.0, 1e-12]) if c["prec"] == "fp64" else 0.0
    c["sort_every"] = rng.choice([10, 0]) if c["prec"] == "mixed" else 10 if c["steps"] > 1 else rng.choice([10, 5, 1])
    return c


# --- inputs ------------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _config(c, **over):
    return dict(metric="ks", a=c["a"], n_r=c["n_r"], n_theta=c["n_theta"], r_min=c["r_min"], r_max=c["r_max"],
                r_absorb=0.9 * c["r_max"], cfl=0.5, precision=c.get("prec", "fp64"), r0=c.get("r0", 0.0),
                h0=c.get("h0", 0.0), n_filter=c.get("n_filter", 0), sort_every=c.get("sort_every", 0),
                iter_tol=c.get("iter_tol", 0.0)) | over


def _momenta(n, theta, g):
    """n isotropic Maxwell-Juttner momenta in an orthonormal frame, (3, n)."""
    u = torch.linspace(0.0, math.sqrt((1.0 + 60.0 * theta) ** 2 - 1.0), 200001, dtype=F8, device=DEV)
    f = u * u * torch.exp(-(torch.sqrt(1.0 + u * u) - 1.0) / theta)
    cdf = torch.cumsum(f, 0)
    mag = u[torch.searchsorted(cdf / cdf[-1], torch.rand(n, generator=g, dtype=F8, device=DEV)).clamp_(max=200000)]
    mag = mag * (1.0 - 1e-6 * torch.rand(n, generator=g, dtype=F8, device=DEV))
    mu = 2.0 * torch.rand(n, generator=g, dtype=F8, device=DEV) - 1.0
    ph = 2.0 * math.pi * torch.rand(n, generator=g, dtype=F8, device=DEV)
    st = torch.sqrt(1.0 - mu * mu)
    return torch.stack([mag * st * torch.cos(ph), mag * st * torch.sin(ph), mag * mu])


def _pieces(n, size=1 << 22):
    return [slice(b, min(n, b + size)) for b in range(0, n, size)]


def _covariant(c, i1, i2, dx1, dx2, uh):
    """Covariant momenta of frame momenta uh at a position, and the weight of unit density there."""
    u, w = torch.empty_like(uh), torch.empty_like(dx1)
    for s in _pieces(dx1.numel()):
        m = _metric(c, i1[s] + dx1[s], i2[s] + dx2[s], clamp=True)
        u[0, s] = uh[0, s] / torch.sqrt(m["H11"]) + m["h13"] / torch.sqrt(m["h33"]) * uh[2, s]
        u[1, s] = torch.sqrt(m["h22"]) * uh[1, s]
        u[2, s] = torch.sqrt(m["h33"]) * uh[2, s]
        w[s] = m["r"] ** (-c.get("power", 0.0)) * m["sh"]
    return u, w


def _particles(c, seed):
    """The initial state of each species, and (q/m, deposit coefficient) of each."""
    g, f = _gen(seed), torch.float32 if c["prec"] == "mixed" else F8
    if c["kind"] == "push":
        n = c["n"]
        x1 = c["n_r"] * (0.05 + 0.9 * torch.rand(n, generator=g, dtype=F8, device=DEV))
        x2 = c["n_theta"] * torch.rand(n, generator=g, dtype=F8, device=DEV)
        i1, i2 = x1.floor().to(torch.int32), x2.floor().to(torch.int32).clamp_(max=c["n_theta"] - 1)
        dx1, dx2 = x1 - i1, x2 - i2
        signs, scale = [1.0], 1.0
    else:
        cells = torch.arange(c["n_r"] * c["n_theta"], device=DEV).repeat_interleave(c["ppc"])
        i1, i2 = (cells % c["n_r"]).to(torch.int32), (cells // c["n_r"]).to(torch.int32)
        del cells
        n = i1.numel()
        dx1, dx2 = (torch.rand(n, generator=g, dtype=F8, device=DEV) for _ in range(2))
        signs, scale = [-1.0, 1.0], 1.0 / c["ppc"]
    out, coef = [], []
    for sign in signs:
        u, w = _covariant(c, i1, i2, dx1, dx2, _momenta(n, c["theta"], g))
        out.append(dict(i1=i1, i2=i2, dx1=dx1.to(f), dx2=dx2.to(f), u1=u[0].to(f), u2=u[1].to(f), u3=u[2].to(f),
                        phi=torch.zeros(n, dtype=f, device=DEV), w=(w * scale).to(f),
                        tag=torch.ones(n, dtype=torch.uint8, device=DEV)))
        rho0, d0 = c.get("rho0", 1.0), c.get("d0", 1.0)
        coef.append((sign / rho0, sign * rho0 / (4.0 * math.pi * d0 * d0)))
    return out, coef


def _pool(c, seed):
    g = _gen(seed + 7919)
    xs = torch.rand(2, POOL_N, generator=g, dtype=F8, device=DEV)
    return torch.cat([xs, _momenta(POOL_N, c["theta"], g), _momenta(POOL_N, c["theta"], g)]).T.contiguous()


def _amplitude(seed):
    return 0.5 + torch.rand(1, generator=_gen(seed), dtype=F8, device=DEV).item()


def _wave(c, seed):
    """A seeded perturbation of B^3 (axisymmetric, so free of divergence), on the stored points."""
    k = torch.rand(3, generator=_gen(seed + 1), dtype=F8, device=DEV)
    x1 = torch.arange(-G, c["n_r"] + G + 1, dtype=F8, device=DEV) + 0.5
    x2 = torch.arange(-G, c["n_theta"] + G + 1, dtype=F8, device=DEV)[:, None] + 0.5
    y1, y2 = x1 / c["n_r"], x2 / c["n_theta"]
    bump = torch.exp(-((y1 - 0.3 - 0.4 * k[0]) / 0.08) ** 2) * torch.sin(math.pi * y2) ** 3
    w = 0.05 * bump * torch.sin(2.0 * math.pi * ((6.0 + 6.0 * k[1]) * y1 + 3.0 * k[2]))
    w[:G] = 0.0
    w[G + c["n_theta"]:] = 0.0
    return w


def _probes(c, seed):
    g, n = _gen(seed), c["n"]
    r = torch.rand(3, n, generator=g, dtype=F8, device=DEV)
    s = torch.empty(6, n, dtype=F8, device=DEV)
    s[0], s[1], s[2] = c["n_r"] * (0.35 + 0.3 * r[0]), c["n_theta"] * (0.35 + 0.3 * r[1]), 0.0
    uh = torch.randn(3, n, generator=g, dtype=F8, device=DEV)
    uh = 0.5 * r[2] * uh / uh.norm(dim=0)
    zero = torch.zeros(n, dtype=F8, device=DEV)
    s[3:] = _covariant(c, s[0], s[1], zero, zero, uh)[0]
    return s, torch.randn(6, n, generator=g, dtype=F8, device=DEV)


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "adjoint":
        sim = P.Sim(_config(c, sort_every=0), [1])
        sim.init_metric()
        sim.init_fields(FIELDS[c["field"]], 1.0)
        s0, v = _probes(c, seed)
        return dict(c=c, sim=sim, s0=s0.requires_grad_(), v=v,
                    b0=torch.tensor(1.0, dtype=F8, requires_grad=True))
    if c["kind"] == "vacuum":
        sim = P.Sim(_config(c), [1])
        sim.init_metric()
        sim.init_fields(FIELDS[c["field"]], _amplitude(seed))
        sim.plane(2).add_(_wave(c, seed).to(sim.tfdtype))
        sim.init_fields(P.FIELD_USER)
        return dict(c=c, sim=sim)
    parts, coef = _particles(c, seed)
    n = parts[0]["i1"].numel()
    over = dict(massless=[0]) if c.get("massless") else {}
    room = 2 * n if c.get("inject") else n
    sim = P.Sim(_config(c, **over), [room] * len(parts))
    sim.init_metric()
    sim.init_fields(FIELDS[c["field"]], 1.0)
    for k, p in enumerate(parts):
        sim.set_particles(k, p, *coef[k])
    st = dict(c=c, sim=sim)
    if c["kind"] == "pic":
        sim.set_keep_prev(False)  # a run without the charge check
    if c.get("host"):
        st["host"] = [{k: torch.empty(v.shape, dtype=v.dtype, pin_memory=True).copy_(v) for k, v in p.items()}
                      for p in parts]
        st["counts"] = [n] * len(parts)
    if c.get("inject"):
        st["pool"], st["calls"], st["room"] = _pool(c, seed), 0, room
    return st


# --- one pass ----------------------------------------------------------------------------------


def _grid_state(sim):
    """The fields and the last step's currents."""
    return {k: sim.plane(p) for k, p in zip(("B1", "B2", "B3", "D1", "D2", "D3", "J1", "J2", "J3"),
                                            (*range(6), *LAST_J))}


def _species(sim, c, k):
    v = sim.species_views(k)
    if c["prec"] == "fp64":
        return {q: v[q] for q in KEYS}
    return {"x1": v["i1"].double().add_(v["dx1"]), "x2": v["i2"].double().add_(v["dx2"]),
            **{q: v[q] for q in KEYS[4:]}}


def _padded(v, n):
    return {k: torch.nn.functional.pad(x, (0, n - x.numel())) for k, x in v.items()}


def run(state):
    c, sim = state["c"], state["sim"]
    if c["kind"] == "adjoint":
        out = P.push_adjoint(sim, state["s0"], state["b0"], 1.0, c["steps"], ckpt_every=c["every"])
        gs, gb = torch.autograd.grad(out, (state["s0"], state["b0"]), state["v"])
        return {"state": out, "grad_state": gs, "grad_b0": gb}
    if c["kind"] == "push":
        for _ in range(c["steps"]):
            sim.push(0)
        return {"0": _species(sim, c, 0)}
    if c["kind"] == "vacuum":
        sim.step(c["steps"])
        return _grid_state(sim)
    if c["host"]:
        state["counts"] = sim.step_host(state["host"], state["counts"])
        return {**_grid_state(sim), **{str(k): {q: v[:m] for q, v in p.items()}
                                       for k, (p, m) in enumerate(zip(state["host"], state["counts"]))}}
    sim.step(c["steps"])
    if c["inject"]:
        sim.inject(SIGMA0, SIGMA_TH, 1.0, state["pool"], 0 if state["calls"] == 0 else -1)
        state["calls"] += 1
    if c["prec"] == "mixed" and c["sort_every"]:
        return _grid_state(sim)
    out = {str(k): _species(sim, c, k) for k in range(2)}
    if c["inject"]:  # as many pairs are added as the plasma asks for: into arrays of one length
        out = {k: _padded(v, state["room"]) for k, v in out.items()}
    return {**_grid_state(sim), **out}


def work(case):
    """Each step reads and writes the state once; a particle's step evaluates the metric twice, a
    field point's the curls and averages of both fields."""
    c = case
    mixed = c.get("prec") == "mixed"
    f, cells = (4 if mixed else 8), (c["n_r"] + 5) * (c["n_theta"] + 5)
    if c["kind"] == "adjoint":
        # forward and reverse: the state, the checkpoints and the cotangents
        n_ck = -(-c["steps"] // c["every"])
        return {"bytes": 48.0 * c["n"] * (4 + 2 * n_ck), "flops": 4500.0 * c["n"] * c["steps"]}
    fields = {"bytes": 24.0 * f * cells, "flops": 130.0 * cells}
    if c["kind"] == "vacuum":
        return {k: c["steps"] * v for k, v in fields.items()}
    one = 9 + 7 * f + 8 + 6 * f  # i1, i2, tag and seven floating values in; cells and six values out
    if c["kind"] == "push":
        return {"bytes": float(c["steps"] * c["n"] * one + 6 * f * cells),
                "flops": c["steps"] * c["n"] * (400.0 if c["massless"] else 700.0)}
    n = 2.0 * c["ppc"] * c["n_r"] * c["n_theta"]
    return {"bytes": c["steps"] * (n * one + fields["bytes"]), "flops": c["steps"] * (n * 760.0 + fields["flops"])}


# --- the same results in 64 bits, from the equations ---------------------------------------------


class _D:
    """A value with its derivatives along x1 and x2."""

    def __init__(self, v, a=0.0, b=0.0):
        self.v, self.a, self.b = v, a, b

    def __add__(self, o):
        o = o if isinstance(o, _D) else _D(o)
        return _D(self.v + o.v, self.a + o.a, self.b + o.b)

    __radd__ = __add__

    def __neg__(self):
        return _D(-self.v, -self.a, -self.b)

    def __sub__(self, o):
        return self + (-o)

    def __rsub__(self, o):
        return -self + o

    def __mul__(self, o):
        o = o if isinstance(o, _D) else _D(o)
        return _D(self.v * o.v, self.a * o.v + self.v * o.a, self.b * o.v + self.v * o.b)

    __rmul__ = __mul__

    def inv(self):
        i = 1.0 / self.v
        return _D(i, -self.a * i * i, -self.b * i * i)

    def sqrt(self):
        s = torch.sqrt(self.v)
        return _D(s, 0.5 * self.a / s, 0.5 * self.b / s)


def _map(c):
    r0 = c.get("r0", 0.0)
    return r0, math.log((c["r_max"] - r0) / (c["r_min"] - r0)) / c["n_r"], math.pi / c["n_theta"]


def _point(c, x1, x2, clamp=False):
    """r, sin and cos of theta, dr/dx1 and dtheta/dx2 at a point."""
    r0, dxi, dth = _map(c)
    e = (c["r_min"] - r0) * torch.exp(x1 * dxi)
    eta, h0 = x2 * dth, c.get("h0", 0.0)
    q = 2.0 * h0 / math.pi ** 2
    th = eta + q * eta * (math.pi - 2.0 * eta) * (math.pi - eta)
    gg = dth * (1.0 + q * (math.pi ** 2 - 6.0 * math.pi * eta + 6.0 * eta * eta))
    gp = dth * dth * q * (12.0 * eta - 6.0 * math.pi)
    if clamp:
        th = th.clamp(1e-5, math.pi - 1e-5)
    s, co = torch.sin(th), torch.cos(th)
    z = torch.zeros_like(e + s)
    return (_D(r0 + e + z, dxi * e + z), _D(s + z, 0.0, co * gg), _D(co + z, 0.0, -s * gg),
            _D(dxi * e + z, dxi * dxi * e + z), _D(gg + z, 0.0, gp + z))


def _metric_d(c, x1, x2, clamp=False):
    """The Kerr-Schild 3-metric, lapse and shift in code units with their derivatives (M = 1)."""
    a = c["a"]
    r, s, co, f, gg = _point(c, x1, x2, clamp)
    s2, r2 = s * s, r * r
    S = r2 + a * a * (co * co)
    z = 2.0 * (r * S.inv())
    A = (r2 + a * a) * (r2 + a * a) - a * a * ((r2 - 2.0 * r + a * a) * s2)
    iS, fi, al2 = S.inv(), f.inv(), (1.0 + z).inv()
    return dict(r=r, s=s, S=S, z=z, A=A, f=f, gg=gg, alpha=al2.sqrt(), beta=z * al2 * fi,
                H11=A * iS * iS * al2 * fi * fi, H13=a * (iS * fi), H22=iS * (gg * gg).inv(), H33=iS * s2.inv(),
                h11=f * f * (1.0 + z), h13=-a * (f * (1.0 + z) * s2), h22=gg * gg * S, h33=A * s2 * iS,
                sht=f * gg * S * (1.0 + z).sqrt())


def _metric(c, x1, x2, clamp=False):
    m = {k: v.v for k, v in _metric_d(c, x1, x2, clamp).items()}
    u = {k: v.v for k, v in zip("rscfg", _point(c, x1, x2))}
    m["sh"] = m["sht"] * (u["s"] if clamp else m["s"])
    return m


def _dt(c):
    x1 = torch.arange(c["n_r"], dtype=F8, device=DEV)[None, :] + 0.5
    x2 = torch.arange(c["n_theta"], dtype=F8, device=DEV)[:, None] + 0.5
    m = _metric(c, x1, x2)
    return 0.5 * (1.0 / (m["alpha"] * torch.sqrt(m["H11"] + m["H22"]) + m["beta"].abs())).min().item()


def _axes(c, s1, s2):
    x1 = torch.arange(-G, c["n_r"] + G + 1, dtype=F8, device=DEV)[None, :] + s1
    x2 = torch.arange(-G, c["n_theta"] + G + 1, dtype=F8, device=DEV)[:, None] + s2
    return x1, x2


def _tables(c):
    """The metric on the four kinds of grid points (0 or 1/2 in x1, x2)."""
    t = {}
    for cls, (s1, s2) in dict(NN=(0, 0), HN=(0.5, 0), NH=(0, 0.5), HH=(0.5, 0.5)).items():
        m = _metric(c, *_axes(c, s1, s2))
        t[cls] = dict(al=m["alpha"], h11=m["h11"], h22=m["h22"], h33=m["h33"], w=0.5 / m["sht"],
                      w13=m["sht"] * m["h13"], wb=m["sht"] * m["sh"] * m["beta"], ish=1.0 / m["sh"])
    return t


def _at(p, di, dj):
    return torch.roll(p, (-dj, -di), (0, 1))


def _potential(c, B0, x1, x2):
    r, s, co, f, gg = _point(c, x1, x2)
    z0 = 0.0 * r
    if c["field"] == "monopole":
        return z0, z0, -B0 * co
    a, s2 = c["a"], s * s
    S = r * r + a * a * (co * co)
    z = 2.0 * (r * S.inv())
    A = (r * r + a * a) * (r * r + a * a) - a * a * ((r * r - 2.0 * r + a * a) * s2)
    h = 0.5 * B0
    return h * a * (z * (2.0 - s2) - 2.0), h * a * (f * (2.0 * z - (1.0 + z) * s2)), h * (A * s2 * S.inv() - 2.0 * a * a * (z * s2))


def _initial_fields(c, B0):
    """B from the discrete curl of A_3 and A_1, D from E_i = d_i A_0."""
    N, rows = c["n_theta"], torch.arange(-G, c["n_theta"] + G + 1, device=DEV)[:, None]
    half, node, inner = (rows >= 0) & (rows < N), (rows >= 0) & (rows <= N), (rows > 0) & (rows < N)
    X = {cls: _axes(c, *s) for cls, s in dict(NN=(0, 0), HN=(0.5, 0), NH=(0, 0.5), HH=(0.5, 0.5)).items()}
    sh = {k: _metric(c, *x)["sh"] for k, x in X.items()}
    zero = torch.zeros_like(sh["NN"])
    x1, x2 = X["NN"]
    lo, up = _potential(c, B0, x1, x2)[2].v, _potential(c, B0, x1, x2 + 1.0)[2].v
    d3 = up - lo
    th = lambda x: x * (math.pi / N) + 2.0 * c.get("h0", 0.0) / math.pi ** 2 * (x * (math.pi / N)) * (  # noqa: E731
        math.pi - 2.0 * x * (math.pi / N)) * (math.pi - x * (math.pi / N))
    sm, df = th(x2 + 1.0) + th(x2), th(x2 + 1.0) - th(x2)
    if c["field"] == "monopole":
        d3 = 2.0 * B0 * torch.sin(0.5 * sm) * torch.sin(0.5 * df) + zero
    B1 = torch.where(half, d3 / sh["NH"], zero)
    B2 = torch.where(inner, -(_potential(c, B0, x1 + 1.0, x2)[2].v - lo) / sh["HN"], zero)
    B3 = zero.clone()
    if c["field"] == "wald":  # A_1(theta_{j+1}) - A_1(theta_j) in product form
        a = c["a"]
        r, f = (_point(c, x1 + 0.5, x2)[q].v for q in (0, 3))
        Sa, Sb = r * r + (a * torch.cos(th(x2))) ** 2, r * r + (a * torch.cos(th(x2 + 1.0))) ** 2
        d1 = -0.5 * B0 * a * f * torch.sin(df) * torch.sin(sm) * (1.0 + 2.0 * r * (r * r - a * a) / (Sa * Sb))
        B3 = torch.where(half, -d1 / sh["HH"], zero)
    D = []
    for cls, rows_of in (("HN", node), ("NH", half), ("NN", inner)):
        m = _metric(c, *X[cls])
        A0, A1, A3 = _potential(c, B0, *X[cls])
        v = ((m["H11"] * A0.a + m["H13"] * m["beta"] * A3.a), m["H22"] * (A0.b - m["beta"] * A1.b),
             (m["H13"] * A0.a + m["H33"] * m["beta"] * A3.a))[len(D)] / m["alpha"]
        D.append(torch.where(rows_of, v, zero))
    return [B1, B2, B3], D


class _Run:
    """A run in 64 bits: the loop of the method on whole planes and particle arrays."""

    def __init__(self, c, B0=1.0):
        self.c, self.dt, self.t = c, _dt(c), _tables(c)
        self.N, self.M, self.nf = c["n_theta"], c["n_r"], c.get("n_filter", 0)
        self.i = torch.arange(-G, self.M + G + 1, device=DEV)[None, :]
        self.j = torch.arange(-G, self.N + G + 1, device=DEV)[:, None]
        self.B, self.D = _initial_fields(c, B0)
        r0, dxi, _ = _map(c)
        x = lambda o: torch.exp((self.i.double() + o) * dxi) * (c["r_min"] - r0)  # noqa: E731
        r_abs = 0.9 * c["r_max"]
        self.k = [(((r0 + x(o) - r_abs) / (c["r_max"] - r_abs)).clamp(0.0, 1.0)) ** 3 for o in (0.0, 0.5)]
        e = x(0.5)
        R = r0 + e
        q = R * R + c["a"] ** 2
        th = _point(c, e, torch.full_like(e, 0.5))
        self.polar = dxi * e * q * torch.sqrt(1.0 + 2.0 * R / q) * (1.0 - th[2].v)
        self.parts, self.coef, self.cursor = [], [], 0
        self.start()

    def start(self):
        f32 = self.c.get("prec") == "mixed"
        self.B, self.D = ([p.float().double() if f32 else p for p in q] for q in (self.B, self.D))
        for q, isB in ((self.B, True), (self.D, False)):
            self.edges(q, isB)
        self.B0, self.D0, self.Bi, self.Di = ([p.clone() for p in q] for q in (self.B, self.D, self.B, self.D))
        self.J0 = [torch.zeros_like(p) for p in self.B]

    def edges(self, F, isB, axis=True):
        """The horizon layer, then the rows across the axes by reflection."""
        N = self.N
        for k, p in enumerate(F):
            p[:, :self.nf + 1 + G] = p[:, self.nf + 1 + G:self.nf + 2 + G].clone()
            if not axis:
                continue
            par, half = (1.0 if k == 0 else -1.0), (k != 1) == isB
            for q in range(1, G + 1):
                if half:
                    p[G - q] = par * p[G + q - 1]
                else:
                    p[G - q], p[G + N + q] = par * p[G + q], par * p[G + N - q]
            if half:
                for q in range(G + 1):
                    p[G + N + q] = par * p[G + N - 1 - q]

    def E(self, B, D):
        t = self.t
        NN, HN, NH, HH = t["NN"], t["HN"], t["NH"], t["HH"]
        a = NN["w13"] * D[2]
        e1 = HN["al"] * (HN["h11"] * D[0] + (a + _at(a, 1, 0)) * HN["w"])
        a, b = HN["w13"] * D[0], HN["wb"] * B[1]
        e3 = NN["al"] * (NN["h33"] * D[2] + (a + _at(a, -1, 0)) * NN["w"]) + (b + _at(b, -1, 0)) * NN["w"]
        e3 = torch.where((self.j == 0) | (self.j == self.N), torch.zeros_like(e3), e3)
        b = HH["wb"] * B[2]
        return e1, NH["al"] * NH["h22"] * D[1] - (b + _at(b, -1, 0)) * NH["w"], e3

    def H(self, B, D):
        t = self.t
        NN, HN, NH, HH = t["NN"], t["HN"], t["NH"], t["HH"]
        a = HH["w13"] * B[2]
        h1 = NH["al"] * (NH["h11"] * B[0] + (a + _at(a, -1, 0)) * NH["w"])
        a, b = NH["w13"] * B[0], NH["wb"] * D[1]
        h3 = HH["al"] * (HH["h33"] * B[2] + (a + _at(a, 1, 0)) * HH["w"]) - (b + _at(b, 1, 0)) * HH["w"]
        b = NN["wb"] * D[2]
        return h1, HN["al"] * HN["h22"] * B[1] + (b + _at(b, 1, 0)) * HN["w"], h3

    def faraday(self, B, E, absorb):
        i, j, M, N, t, dt = self.i, self.j, self.M, self.N, self.t, self.dt
        out = [p.clone() for p in B]
        half, c0, c1 = (j >= 0) & (j < N), (i >= 0) & (i <= M), (i >= 0) & (i < M)
        for k, (where, d) in enumerate((
                (half & c0, -(_at(E[2], 0, 1) - E[2]) * t["NH"]["ish"]),
                ((j >= 1) & (j < N) & c1, (_at(E[2], 1, 0) - E[2]) * t["HN"]["ish"]),
                (half & c1, -((_at(E[1], 1, 0) - E[1]) - (_at(E[0], 0, 1) - E[0])) * t["HH"]["ish"]))):
            out[k] = torch.where(where, out[k] + dt * d, out[k])
            if absorb:
                kk = self.k[0] if k == 0 else self.k[1]
                out[k] = torch.where((j >= 0) & (j <= N), out[k] - kk * (out[k] - self.Bi[k]), out[k])
        return out

    def ampere(self, D, H, J, absorb):
        i, j, M, N, t, dt, fp = self.i, self.j, self.M, self.N, self.t, self.dt, 4.0 * math.pi
        dn = H[2] - _at(H[2], 0, -1)
        d1 = torch.where(j == 0, (H[2] - fp * J[0]) / self.polar,
                         torch.where(j == N, (-_at(H[2], 0, -1) - fp * J[0]) / self.polar,
                                     (dn - fp * J[0]) * t["HN"]["ish"]))
        d2 = (-(H[2] - _at(H[2], -1, 0)) - fp * J[1]) * t["NH"]["ish"]
        d3 = ((H[1] - _at(H[1], -1, 0)) - (H[0] - _at(H[0], 0, -1)) - fp * J[2]) * t["NN"]["ish"]
        c0, c1, half = (i >= 0) & (i <= M), (i >= 0) & (i < M), (j >= 0) & (j < N)
        out = []
        for k, (where, d) in enumerate((((j >= 0) & (j <= N) & c1, d1), (half & c0, d2), ((j >= 1) & (j < N) & c0, d3))):
            p = torch.where(where, D[k] + dt * d, D[k])
            if absorb:
                kk = self.k[1] if k == 0 else self.k[0]
                p = torch.where((j >= 0) & (j <= N), p - kk * (p - self.Di[k]), p)
            out.append(p)
        return out

    def fields_at(self, Bn, D, x1, x2):
        out = []
        for p, o1, o2 in zip((*Bn, *D), (0, .5, .5, .5, 0, 0), (.5, 0, .5, 0, .5, 0)):
            y1, y2 = x1 - o1, x2 - o2
            f1, f2 = y1.detach().floor(), y2.detach().floor()
            w1, w2 = y1 - f1, y2 - f2
            k = (f2.long() + G) * p.shape[1] + f1.long() + G
            q = p.reshape(-1)
            out.append((1 - w2) * ((1 - w1) * q[k] + w1 * q[k + 1]) +
                       w2 * ((1 - w1) * q[k + p.shape[1]] + w1 * q[k + p.shape[1] + 1]))
        return out[:3], out[3:]

    def orbit(self, x1, x2, u, F, qm, m2, n_iter, scale=1.0):
        """The move of particles: new offsets from x^n, momenta, and a function for dphi/dt."""
        c, dt = self.c, self.dt
        m = _metric_d(c, x1, x2, clamp=True)
        v = {k: q.v for k, q in m.items()}
        sH, s22, s33 = torch.sqrt(v["H11"]), torch.sqrt(v["h22"]), torch.sqrt(v["h33"])
        if m2:
            Bv, Dv = self.fields_at(*F, x1, x2)
            hat = lambda A: (scale * A[0] / sH, scale * s22 * A[1], scale * (v["h13"] / s33 * A[0] + s33 * A[2]))  # noqa: E731
            Bh, Dh = hat(Bv), hat(Dv)

        def kick(u):
            if not m2:
                return u
            e = 0.25 * qm * dt * v["alpha"]
            w = (sH * (u[0] - v["h13"] / v["h33"] * u[2]), u[1] / s22, u[2] / s33)
            w = [w[q] + e * Dh[q] for q in range(3)]
            ig = 1.0 / torch.sqrt(1.0 + w[0] ** 2 + w[1] ** 2 + w[2] ** 2)
            t = [e * Bh[q] * ig for q in range(3)]
            sf = 2.0 / (1.0 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2)
            cr = lambda p, q: (p[1] * q[2] - p[2] * q[1], p[2] * q[0] - p[0] * q[2], p[0] * q[1] - p[1] * q[0])  # noqa: E731
            p = [w[q] + x for q, x in enumerate(cr(w, t))]
            w = [w[q] + sf * x + e * Dh[q] for q, x in enumerate(cr(p, t))]
            return (w[0] / sH + v["h13"] / s33 * w[2], s22 * w[1], s33 * w[2])

        u = kick(u)
        t = [u[0], u[1]]
        for _ in range(n_iter):
            b = (0.5 * (t[0] + u[0]), 0.5 * (t[1] + u[1]), u[2])
            gam = torch.sqrt(m2 + v["H11"] * b[0] ** 2 + v["H22"] * b[1] ** 2 + v["H33"] * b[2] ** 2 + 2 * v["H13"] * b[0] * b[2])
            t = [u[q] - dt * gam * g("alpha") + dt * b[0] * g("beta") - 0.5 * dt * v["alpha"] / gam * (
                g("H11") * b[0] ** 2 + g("H22") * b[1] ** 2 + g("H33") * b[2] ** 2 + 2 * g("H13") * b[0] * b[2])
                for q, g in enumerate((lambda k: m[k].a, lambda k: m[k].b))]
        u = kick((t[0], t[1], u[2]))

        def rate(y1, y2):
            o = _metric(c, y1, y2, clamp=True)
            gam = torch.sqrt(m2 + o["H11"] * u[0] ** 2 + o["H22"] * u[1] ** 2 + o["H33"] * u[2] ** 2 + 2 * o["H13"] * u[0] * u[2])
            ag = o["alpha"] / gam
            return (ag * (o["H11"] * u[0] + o["H13"] * u[2]) - o["beta"], ag * o["H22"] * u[1],
                    ag * (o["H13"] * u[0] + o["H33"] * u[2]))

        d = (torch.zeros_like(x1), torch.zeros_like(x2))
        for _ in range(n_iter):
            d = [dt * q for q in rate(x1 + 0.5 * d[0], x2 + 0.5 * d[1])[:2]]
        return d, u, rate

    def move(self, p, Bn, qm, qc, m2, J):
        """One species through one step; J (if given) takes its currents."""
        N, M, dt, NX = self.N, self.M, self.dt, self.B[0].shape[1]
        live = torch.nonzero(p["tag"] == 1).reshape(-1)
        p["tag"] = torch.where(p["tag"] == 1, p["tag"], torch.zeros_like(p["tag"]))
        for s in _pieces(live.numel(), 1 << 21):
            k = live[s]
            i1, i2, dx1, dx2 = (p[q][k] for q in KEYS[:4])
            d, u, _ = self.orbit(i1 + dx1, i2 + dx2, [p[q][k] for q in ("u1", "u2", "u3")], (Bn, self.D), qm, m2, 10)
            t1, t2 = dx1 + d[0], dx2 + d[1]
            f1, f2 = t1.floor(), t2.floor()
            j1, j2, e1, e2 = i1 + f1.int(), i2 + f2.int(), t1 - f1, t2 - f2
            flip = (j2 < 0) | (j2 >= N)
            e2, j2 = torch.where(flip, 1.0 - e2, e2), j2.clamp(0, N - 1)
            u = (u[0], torch.where(flip, -u[1], u[1]), u[2])
            xa1, xa2, xb1, xb2 = i1 + dx1, i2 + dx2, j1 + e1, j2 + e2
            m1, mm2 = i1 + 0.5 * (dx1 + (j1 - i1) + e1), i2 + 0.5 * (dx2 + (j2 - i2) + e2)
            o = _metric(self.c, m1, mm2, clamp=True)
            gam = torch.sqrt(m2 + o["H11"] * u[0] ** 2 + o["H22"] * u[1] ** 2 + o["H33"] * u[2] ** 2 + 2 * o["H13"] * u[0] * u[2])
            v3 = o["alpha"] / gam * (o["H13"] * u[0] + o["H33"] * u[2])
            for q, v in zip(("i1", "i2", "dx1", "dx2", "u1", "u2", "u3"), (j1, j2, e1, e2, *u)):
                p[q][k] = v
            p["phi"][k] += dt * v3
            p["tag"][k] = torch.where((j1 < 0) | (j1 >= M), 2, 1).to(torch.uint8)
            if J is None:
                continue
            q = qc * p["w"][k]
            lo1, hi1 = torch.minimum(i1, j1).double() + 1.0, torch.maximum(i1, j1).double()
            lo2, hi2 = torch.minimum(i2, j2).double() + 1.0, torch.maximum(i2, j2).double()
            xr1 = torch.minimum(lo1, torch.maximum(hi1, 0.5 * (xa1 + xb1)))
            xr2 = torch.minimum(lo2, torch.maximum(hi2, 0.5 * (xa2 + xb2)))
            add = lambda c, n, v: J[c].view(-1).index_add_(0, n, v)  # noqa: E731
            for ci, cj, y1, y2, z1, z2 in ((i1, i2, xa1, xa2, xr1, xr2), (j1, j2, xr1, xr2, xb1, xb2)):
                F1, F2 = q * (z1 - y1) / dt, q * (z2 - y2) / dt
                W1, W2 = 0.5 * (y1 + z1) - ci, 0.5 * (y2 + z2) - cj
                n = (cj.long() + G) * NX + ci.long() + G
                add(0, n, F1 * (1 - W2)), add(0, n + NX, F1 * W2), add(1, n, F2 * (1 - W1)), add(1, n + 1, F2 * W1)
            c1, c2 = m1.floor(), mm2.floor()
            w1, w2, qv = m1 - c1, mm2 - c2, q * v3
            n = (c2.long() + G) * NX + c1.long() + G
            for o, w in ((0, (1 - w1) * (1 - w2)), (1, w1 * (1 - w2)), (NX, (1 - w1) * w2), (NX + 1, w1 * w2)):
                add(2, n + o, qv * w)

    def smooth(self, J):
        """n_f passes of the binomial filter on the grid extended across the axes by reflection."""
        N = self.N
        for c, half, par in ((0, False, 1.0), (1, True, -1.0), (2, False, 1.0)):
            p = J[c][G:G + (N if half else N + 1)].clone()
            if not half:
                p[0], p[N] = 2.0 * p[0], 2.0 * p[N]
            for _ in range(self.nf):
                z = torch.zeros_like(p[:, :1])
                p = torch.cat([z, p[:, :-1]], 1) + 2.0 * p + torch.cat([p[:, 1:], z], 1)
                lo, hi = (p[:1], p[-1:]) if half else (p[1:2], p[-2:-1])
                p = (torch.cat([par * lo, p[:-1]]) + 2.0 * p + torch.cat([p[1:], par * hi])) / 16.0
            if not half:
                p[0], p[N] = 0.5 * p[0], 0.5 * p[N]
            J[c].zero_()
            J[c][G:G + p.shape[0]] = p

    def sort(self, p):
        tr = tt = 16
        key = ((p["i2"] // tt) * (-(-self.M // tr)) + p["i1"] // tr).long() * (tr * tt) + (p["i2"] % tt) * tr + p["i1"] % tr
        key = torch.where(p["tag"] == 1, key, torch.full_like(key, 1 << 40))
        o = torch.sort(key, stable=True).indices[:int((p["tag"] == 1).sum())]
        return {k: v[o] for k, v in p.items()}

    def step(self, sort_now):
        Bm, Dm = ([0.5 * (x + y) for x, y in zip(q0, q)] for q0, q in ((self.B0, self.B), (self.D0, self.D)))
        Bn = self.faraday(Bm, self.E(self.B, Dm), False)
        self.edges(Bn, True)
        if sort_now:
            self.parts = [self.sort(p) for p in self.parts]
        J = [torch.zeros_like(p) for p in self.B]
        for p, (qm, qc) in zip(self.parts, self.coef):
            self.move(p, Bn, qm, qc, 1.0, J)
        if self.nf:
            self.smooth(J)
        E, H = self.E(Bn, self.D), self.H(Bn, self.D)
        B = self.faraday(self.B, E, True)
        self.edges(B, True)
        Dh = self.ampere(Dm, H, [0.5 * (x + y) for x, y in zip(self.J0, J)], False)
        self.edges(Dh, False, axis=False)
        D = self.ampere(self.D, self.H(B, Dh), J, True)
        self.edges(D, False)
        self.B0, self.D0, self.B, self.D, self.J0 = self.B, self.D, B, D, J

    def inject(self, pool):
        """One pair in each cell whose magnetization is above the threshold."""
        c, M, N = self.c, self.M, self.N
        x1 = torch.arange(M, dtype=F8, device=DEV)[None, :] + 0.5
        x2 = torch.arange(N, dtype=F8, device=DEV)[:, None] + 0.5
        m = _metric(c, x1, x2)
        w = torch.zeros(M * N, dtype=F8, device=DEV)
        for p in self.parts:
            k = torch.nonzero(p["tag"] == 1).reshape(-1)
            w.index_add_(0, p["i2"][k].long() * M + p["i1"][k].long(), p["w"][k].abs())
        cut = lambda q: q[G:G + N, G:G + M]  # noqa: E731
        b1 = 0.5 * (cut(self.B[0]) + cut(_at(self.B[0], 1, 0)))
        b2 = 0.5 * (cut(self.B[1]) + cut(_at(self.B[1], 0, 1)))
        b3 = cut(self.B[2])
        bb = m["h11"] * b1 ** 2 + m["h22"] * b2 ** 2 + m["h33"] * b3 ** 2 + 2.0 * m["h13"] * b1 * b3
        n = w.view(N, M) / m["sh"]
        cells = torch.nonzero((SIGMA0 * bb > SIGMA_TH * n).reshape(-1)).reshape(-1)
        wp = (0.5 * (SIGMA0 / SIGMA_TH * bb - n) * m["sh"]).reshape(-1)[cells]
        r = pool[(self.cursor + torch.arange(cells.numel(), device=DEV)) % POOL_N]
        self.cursor += cells.numel()
        i1, i2 = (cells % M).int(), (cells // M).int()
        one = torch.ones_like(wp)
        for q, p in enumerate(self.parts):
            u, _ = _covariant(c, i1, i2, r[:, 0].contiguous(), r[:, 1].contiguous(), r[:, 2 + 3 * q:5 + 3 * q].T.contiguous())
            new = dict(i1=i1, i2=i2, dx1=r[:, 0], dx2=r[:, 1], u1=u[0], u2=u[1], u3=u[2], phi=0.0 * one, w=wp,
                       tag=one.to(torch.uint8))
            self.parts[q] = {k: torch.cat([p[k], new[k]]) for k in KEYS}


def _read(c, parts):
    """The outputs of a run for its particles (whole numbers have no 64-bit value of their own)."""
    if c["prec"] == "fp64":
        return {str(k): {q: (None if q in ("i1", "i2", "tag") else p[q]) for q in KEYS} for k, p in enumerate(parts)}
    return {str(k): {"x1": p["i1"] + p["dx1"], "x2": p["i2"] + p["dx2"], **{q: p[q] for q in KEYS[4:9]}, "tag": None}
            for k, p in enumerate(parts)}


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "adjoint":
        if c["n"] * c["steps"] > 7000000:
            return None
        r = _Run(c)
        s0, v = _probes(c, seed)
        s0.requires_grad_()
        b0 = torch.ones((), dtype=F8, device=DEV, requires_grad=True)
        x1, x2, phi, u = s0[0], s0[1], s0[2], (s0[3], s0[4], s0[5])

        def one(x1, x2, phi, u0, u1, u2, b0):
            d, u, rate = r.orbit(x1, x2, (u0, u1, u2), (r.B, r.D), 1.0, 1.0, 9, scale=b0)
            return x1 + d[0], x2 + d[1], phi + r.dt * rate(x1 + 0.5 * d[0], x2 + 0.5 * d[1])[2], *u

        for _ in range(c["steps"]):
            x1, x2, phi, *u = torch.utils.checkpoint.checkpoint(one, x1, x2, phi, *u, b0, use_reentrant=False)
        out = torch.stack([x1, x2, phi, *u])
        gs, gb = torch.autograd.grad(out, (s0, b0), v)
        return {"state": out.detach(), "grad_state": gs, "grad_b0": gb}
    with torch.no_grad():
        if c["kind"] == "vacuum":
            r = _Run(c, _amplitude(seed))
            f32 = c["prec"] == "mixed"
            w = _wave(c, seed)
            r.B[2] = (r.B[2].float() + w.float()).double() if f32 else r.B[2] + w
            r.start()
            for _ in range(c["steps"]):
                r.step(False)
        else:
            size = c["n"] if c["kind"] == "push" else 2 * c["ppc"] * c["n_r"] * c["n_theta"]
            if size * c["steps"] > 200000000:
                return None
            r = _Run(c)
            parts, r.coef = _particles(c, seed)
            r.parts = [{k: v.double() if v.is_floating_point() else v.clone() for k, v in p.items()} for p in parts]
            del parts
            if c["kind"] == "push":
                for _ in range(c["steps"]):
                    r.move(r.parts[0], r.B, *r.coef[0], 0.0 if c["massless"] else 1.0, None)
                return _read(c, r.parts)
            for k in range(c["steps"]):
                r.step(c["sort_every"] > 0 and k % c["sort_every"] == 0)
            if c["inject"]:
                r.inject(_pool(c, seed))
                r.parts = [_padded(p, c["ppc"] * c["n_r"] * c["n_theta"] * 2) for p in r.parts]
        out = dict(zip(("B1", "B2", "B3", "D1", "D2", "D3", "J1", "J2", "J3"), (*r.B, *r.D, *r.J0)))
        if c["kind"] == "vacuum" or (c["prec"] == "mixed" and c["sort_every"]):
            return out
        return {**out, **_read(c, r.parts)}
