"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one of

  step      one context advances a few time steps (pf_step) and its new state is read
            (phi, velocity, zero-mean pressure): what every simulation does;
  batch     the same for many uneven 2D drops advanced together (pf_batch_step);
  solve     one variable-density pressure solve (pf_poisson_solve) on device arrays;
  rhs       the stage right-hand sides alone (pf_eval_rhs) on device arrays;
  adjoint   the transposed Jacobian of one float64 step (pf_step_adjoint): a link of a
            checkpointed gradient.

Inputs are a drop (or the standing wave between walls) in a seeded divergence-free flow of
about a fifth of the capillary velocity, as it is met in the middle of a run. Mixed-precision
contexts store phi and u in float32, so their inputs are float32 values and their outputs are
returned in float32. `exact` is a plain float64 torch restatement of the same discrete method
(pressure by FFT-preconditioned CG to rounding, adjoint by autograd).
"""
from __future__ import annotations

import math
import random

import torch

# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
_STEP = dict(kind="step", dim=2, nx=64, ny=64, nz=1, precision="fp64", model="cdi", force="eb",
             momentum="advective", scheme="rk4", wall=False, ratio=10.0, rtol=1e-12, graph=False,
             steps=1)


def _case(name=None, **kw):
    c = dict(_STEP, **kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest run anyone makes: the 64^2 static drop in float64, host-driven (the default)
        _case("step_64x64_fp64", ratio=1.0, steps=4),
        # density ratio 1000 drop, ACDI, mixed precision, one graph per step
        _case("step_256x256_r1000_acdi_mixed_graph", nx=256, ny=256, precision="mixed",
              model="acdi", ratio=1000.0, graph=True, steps=4),
        # the walled standing wave study in float64
        _case("wave_128x128_fp64", nx=128, ny=128, wall=True, ratio=1.0, steps=2),
        # a rectangular box off the powers of two, source-form phase field and CSF force
        _case("step_200x136_isodi_csf_fp64_graph", nx=200, ny=136, model="isodi", force="csf",
              graph=True),
        # odd cell counts, forward Euler
        _case("step_61x45_fe_fp64", nx=61, ny=45, scheme="fe"),
        # a parameter study: many uneven 2D drops at once
        _case("batch_32_mixed_graph", kind="batch", count=32, manifest=20261203,
              precision="mixed", rtol=1e-10, graph=True, steps=2),
        # one link of a checkpointed gradient of the 256^2 oscillating drop
        _case("adjoint_256x256_fp64", kind="adjoint", nx=256, ny=256),
        # 3D mixed precision as in the README, host-driven
        _case("step_128x128x128_acdi_mixed", dim=3, nx=128, ny=128, nz=128, precision="mixed",
              model="acdi", rtol=1e-10, steps=2),
        # a rectangular 3D box off the powers of two, conservative momentum transport
        _case("step_160x120x72_consistent_mixed_graph", dim=3, nx=160, ny=120, nz=72,
              precision="mixed", momentum="consistent", ratio=1000.0, rtol=1e-10, graph=True),
        # 3D in float64, the reference precision
        _case("step_96x96x96_fp64_graph", dim=3, nx=96, ny=96, nz=96, graph=True),
        # a pressure solve alone, in a caller's own loop
        _case("solve_192x160x96_mixed", kind="solve", dim=3, nx=192, ny=160, nz=96,
              precision="mixed", rtol=1e-10),
        # the largest: the 384^3 oscillating drop of the benchmark
        _case("step_384x384x384_acdi_mixed_graph", dim=3, nx=384, ny=384, nz=384,
              precision="mixed", model="acdi", rtol=1e-10, graph=True),
    ]


def _sides(rng, k, lo, hi, count):
    """`count` sides m 2^k, m spread over [lo, hi] by its logarithm (m odd or even)."""
    return [int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) << k
            for _ in range(count)]


def _sides2(rng):
    """2D sides from 20 to 512: any count at the small end, multiples of 16 at the large one
    (the study manifest's granularity)."""
    k = rng.randint(0, 4)
    return _sides(rng, k, 20, 40 if k < 4 else 32, 2)


def draw(rng):
    kind = rng.choice(["step2", "step2", "step2", "batch", "adjoint", "step3", "step3", "solve2",
                       "solve3", "rhs"])
    ratio = rng.choice([1.0, 10.0, 1000.0])
    precision = rng.choice(["fp64", "mixed"])
    rtol = 1e-12 if precision == "fp64" else 1e-10
    graph = rng.random() < 0.5
    if kind == "step2":
        nx, ny = _sides2(rng)
        if rng.random() < 0.2:
            return _case(nx=nx, ny=ny, wall=True, ratio=1.0, graph=graph)
        momentum = "consistent" if rng.random() < 0.2 else "advective"
        model = "cdi" if momentum == "consistent" else rng.choice(["cdi", "acdi", "sb", "isodi"])
        return _case(nx=nx, ny=ny, precision=precision, model=model, ratio=ratio, rtol=rtol,
                     force=rng.choice(["eb", "eb", "csf", "lcsf"]), momentum=momentum,
                     scheme=rng.choice(["rk4", "rk4", "fe"]), graph=graph)
    if kind == "batch":
        return _case(kind="batch", count=rng.randint(5, 24), manifest=rng.randrange(1 << 30),
                     precision="mixed", rtol=1e-10, graph=rng.random() < 0.7)
    if kind == "adjoint":
        n = _sides(rng, rng.randint(2, 4), 12, 20, 1)[0]
        return _case(kind="adjoint", nx=n, ny=n, ratio=rng.choice([1.0, 10.0]))
    if kind == "solve2":
        nx, ny = _sides2(rng)
        return _case(kind="solve", nx=nx, ny=ny, ratio=ratio)
    nx, ny, nz = _sides(rng, 3 if precision == "fp64" else rng.choice([3, 4]), 5, 14, 3)
    if kind == "solve3":
        return _case(kind="solve", dim=3, nx=nx, ny=ny, nz=nz, precision=precision, rtol=rtol,
                     ratio=rng.choice([1.0, 10.0]))
    momentum = "consistent" if rng.random() < 0.25 else "advective"
    model = "cdi" if momentum == "consistent" else rng.choice(["cdi", "acdi", "acdi", "sb"])
    return _case(kind="rhs" if kind == "rhs" else "step", dim=3, nx=nx, ny=ny, nz=nz,
                 precision=precision, model=model, momentum=momentum, rtol=rtol,
                 ratio=rng.choice([1.0, 10.0]),
                 graph=graph)


# ---------------------------------------------------------------------------------------------
# parameters and inputs
# ---------------------------------------------------------------------------------------------
def _params(c):
    """The parameter set of a step / solve / rhs / adjoint case (eps = dx, dt half the smaller
    of the capillary and viscous limits, the viscosity ratio ten at most)."""
    dim, n = c["dim"], (c["nx"], c["ny"], c["nz"])
    if c["wall"]:
        L, nu = 2.0 * math.pi, 0.064720863
        p = dict(L=L, sigma=2.0, rho_in=1.0, rho_out=1.0, mu_in=nu, mu_out=nu, eps=L / 32,
                 R=0.5 * c["ny"] * L / c["nx"], wall_y=1, shape="wave", pert_mode=1,
                 pert_amp=0.02)
    else:
        mu = 0.1 if c["ratio"] == 1.0 else 0.01
        p = dict(L=1.0, sigma=1.0, rho_in=10.0, rho_out=10.0 / c["ratio"], mu_in=mu,
                 mu_out=mu / min(c["ratio"], 10.0), eps=1.0 / c["nx"], wall_y=0, shape="drop",
                 R=0.25 * min(n[:dim]) / c["nx"])
    h = p["L"] / c["nx"]
    nu = max(p["mu_in"] / p["rho_in"], p["mu_out"] / p["rho_out"])
    cap = math.sqrt((p["rho_in"] + p["rho_out"]) * h ** 3 / (4.0 * math.pi * p["sigma"]))
    dt = 0.5 * min(cap, h * h / (2.0 * dim * nu))
    if c["wall"]:
        dt = min(0.003, dt)
    p.update(dim=dim, n=n, precision=c["precision"], model=c["model"], force=c["force"],
             momentum=c["momentum"], scheme=c["scheme"], dt=dt, delta_n=1e-12,
             gamma_fixed=0.1 if c["kind"] == "adjoint" else 0.0, poisson_rtol=c["rtol"],
             poisson_maxit=400, use_graph=int(c["graph"]))
    return p


def _batch_params(c):
    """Uneven drops: N in {64, 80, ..., 512}, R in [0.15, 0.3], log10 La in [2, 5], density
    ratio in {1, 10, 1000} (the ranges of the library's seeded study manifest)."""
    r, out = random.Random(c["manifest"]), []
    for _ in range(c["count"]):
        n, R = 16 * r.randint(4, 32), r.uniform(0.15, 0.3)
        ratio = r.choice([1.0, 10.0, 1000.0])
        p = _params(dict(c, kind="step", nx=n, ny=n, ratio=ratio))
        mu = math.sqrt(2.0 * R / 10.0 ** r.uniform(2.0, 5.0))
        h = 1.0 / n
        cap = math.sqrt((1.0 + 1.0 / ratio) * h ** 3 / (4.0 * math.pi))
        p.update(R=R, rho_in=1.0, rho_out=1.0 / ratio, mu_in=mu, mu_out=mu,
                 dt=0.5 * min(cap, h * h / (4.0 * mu * ratio)))
        out.append(p)
    return out


def _inputs(p, seed):
    """(phi, [u, v(, w)]): a slightly deformed drop off the box centre (or the wave) in a
    divergence-free flow of a few modes, float64 on the GPU."""
    r = random.Random(seed)
    dim, n = p["dim"], p["n"]
    h = p["L"] / n[0]
    shape = tuple(reversed(n[:dim]))
    dev = torch.device("cuda")

    def axis(d, off):
        v = [1] * dim
        v[dim - 1 - d] = n[d]
        return ((torch.arange(n[d], dtype=torch.float64, device=dev) + off) * h).reshape(v)

    size = [n[d] * h for d in range(dim)]
    if p["wall_y"]:
        a, s = 0.01 + 0.02 * r.random(), 2.0 * math.pi * r.random()
        yi = p["R"] * (1.0 - a * torch.cos(2.0 * math.pi * axis(0, 0.5) / size[0] + s))
        phi = 0.5 * (1.0 + torch.tanh((yi - axis(1, 0.5)) / (2.0 * p["eps"])))
    else:
        x = [axis(d, 0.5) - size[d] * (0.5 + 0.04 * (r.random() - 0.5)) for d in range(dim)]
        rad = torch.sqrt(sum(v * v for v in x))
        defo = sum((0.03 + 0.03 * r.random()) * v * v for v in x[:-1]) / (rad * rad + h * h)
        phi = 0.5 * (1.0 + torch.tanh((p["R"] * (1.0 + defo) - rad) / (2.0 * p["eps"])))
    phi = phi.expand(shape).contiguous()

    def potential(axes):   # periodic in each axis; zero on the walls where there are any
        out = torch.zeros(shape, dtype=torch.float64, device=dev)
        for _ in range(3):
            t = torch.ones([1] * dim, dtype=torch.float64, device=dev)
            for d in range(dim):
                k, s = r.choice([1, 2]), 2.0 * math.pi * r.random()
                y = axis(d, 0.0 if d in axes else 0.5)
                wall = p["wall_y"] and d == 1
                t = t * (torch.sin(math.pi * k * y / size[d]) if wall else
                         torch.sin(2.0 * math.pi * k * y / size[d] + s))
            out = out + (0.5 + r.random()) * t
        return out

    def up(a, d):
        return (torch.roll(a, -1, dim - 1 - d) - a) / h

    # discrete curl of edge potentials: the discrete divergence is zero to rounding
    a01 = potential((0, 1))
    u = [up(a01, 1), -up(a01, 0)]
    if dim == 3:
        a12, a02 = potential((1, 2)), potential((0, 2))
        u = [u[0] + up(a02, 2), u[1] + up(a12, 2), -up(a02, 0) - up(a12, 1)]
    amp = 0.2 * math.sqrt(p["sigma"] / (p["rho_in"] * p["R"])) * (0.75 + 0.5 * r.random())
    top = max(float(v.abs().max()) for v in u)
    u = [v * (amp / top) for v in u]
    if p["wall_y"]:
        u[1][0] = 0.0
    if p["precision"] == "mixed":
        phi, u = phi.float().double(), [v.float().double() for v in u]
    return phi, u


def _cells(p):
    return p["n"][0] * p["n"][1] * p["n"][2]


def _gamma(u):
    return max(float(v.abs().max()) for v in u)


def _rhs_field(p, phi, u):
    """A right-hand side of the pressure equation as a step meets it: the divergence of a
    velocity with an interfacial part that is not solenoidal, over dt."""
    dim, h = p["dim"], p["L"] / p["n"][0]
    f = [v + 0.3 * v.abs().max() * torch.roll(phi, d + 1, dim - 1) * (1.0 - phi)
         for d, v in enumerate(u)]
    return sum((torch.roll(v, -1, dim - 1 - d) - v) / h for d, v in enumerate(f)) / p["dt"]


# ---------------------------------------------------------------------------------------------
# running them
# ---------------------------------------------------------------------------------------------
def _load(pf, ctx, phi, u):
    for name, v in zip(("phi", "u", "v", "w"), [phi] + u):
        pf.pf_set_field(ctx, pf.FIELDS[name], v.contiguous().data_ptr())


def _state(pf, ctx, p):
    """phi and the velocity in their storage type (one array, components first) and the
    zero-mean pressure."""
    n, dim = _cells(p), p["dim"]
    dtype = torch.float32 if p["precision"] == "mixed" else torch.float64
    raw = torch.empty(pf.pf_state_bytes(ctx), dtype=torch.uint8, device="cuda")
    pf.pf_get_state(ctx, raw.data_ptr())
    pr = torch.empty(n, dtype=torch.float64, device="cuda")
    pf.pf_get_field(ctx, pf.FIELDS["p"], pr.data_ptr())
    width = (1 + dim) * n * (4 if dtype == torch.float32 else 8)
    return raw[:width].view(dtype).view(1 + dim, n), pr.to(dtype)


def prepare(case, seed):
    import paper_2205_05835_gb300 as pf

    kind = case["kind"]
    if kind == "batch":
        plist = _batch_params(case)
        b = pf.Batch(plist)
        for i, p in enumerate(plist):
            _load(pf, pf.pf_batch_context(b.b, i), *_inputs(p, seed * 1000 + i))
        return dict(pf=pf, kind=kind, p=plist, batch=b, steps=case["steps"])
    p = _params(case)
    phi, u = _inputs(p, seed)
    sim = pf.Simulation(p)
    _load(pf, sim.ctx, phi, u)
    s = dict(pf=pf, kind=kind, p=p, sim=sim, steps=case["steps"])
    if kind == "solve":
        s["rhs"] = _rhs_field(p, phi, u).reshape(-1).contiguous()
    elif kind == "rhs":
        s["gamma"] = _gamma(u)
    elif kind == "adjoint":
        from paper_2205_05835_gb300.adjoint import Adjoint

        s["adj"] = Adjoint(sim)
        s["state0"] = sim.state_tensor()
        s["lam"] = _cotangent(p, seed)
    return s


def _cotangent(p, seed):
    """Cotangent of the state after the step: smooth fields of another seed."""
    phi, u = _inputs(p, seed + 7777)
    return torch.stack([phi - phi.mean()] + u).reshape(-1).contiguous()


def run(s):
    pf, kind, p = s["pf"], s["kind"], s["p"]
    if kind == "batch":
        s["batch"].step(s["steps"])
        got = [_state(pf, pf.pf_batch_context(s["batch"].b, i), q) for i, q in enumerate(p)]
        return [torch.cat([f.reshape(-1) for f, _ in got]), torch.cat([q for _, q in got])]
    sim = s["sim"]
    if kind == "step":
        sim.step(s["steps"])
        f, pr = _state(pf, sim.ctx, p)
        return [f[0], f[1:], pr]
    n = _cells(p)
    if kind == "solve":
        x = torch.zeros(n, dtype=torch.float64, device="cuda")
        pf.pf_poisson_solve(sim.ctx, s["rhs"].data_ptr(), x.data_ptr())
        return x.float() if p["precision"] == "mixed" else x
    if kind == "rhs":
        kphi = torch.empty(n, dtype=torch.float64, device="cuda")
        ku = torch.empty(p["dim"] * n, dtype=torch.float64, device="cuda")
        pf.pf_eval_rhs(sim.ctx, s["gamma"], kphi.data_ptr(), ku.data_ptr())
        return [kphi.float(), ku.float()] if p["precision"] == "mixed" else [kphi, ku]
    lam = s["lam"].clone()
    g = torch.zeros(5, dtype=torch.float64, device="cuda")
    s["adj"].step(s["state0"], lam, g)
    return [lam, g]


def work(case):
    """State (or operands) in and results out once; stage arithmetic of about 250 operations a
    cell and one pass of the pressure operator, in each of the stages."""
    ps = _batch_params(case) if case["kind"] == "batch" else [_params(case)]
    out = {"bytes": 0, "flops": 0}
    for p in ps:
        n, dim, w = _cells(p), p["dim"], 4 if p["precision"] == "mixed" else 8
        state = n * ((1 + dim) * w + 8)
        stages = 4 if p["scheme"] == "rk4" else 1
        if case["kind"] in ("step", "batch"):
            b, f = 2 * state, case["steps"] * stages * 270 * n
        elif case["kind"] == "solve":
            b, f = n * (w + 16), 20 * n
        elif case["kind"] == "rhs":
            b, f = n * (1 + dim) * (w + 8), 250 * n
        else:
            b, f = state + 2 * (1 + dim) * 8 * n, 3 * stages * 270 * n
        out["bytes"] += b
        out["flops"] += f
    return out


# ---------------------------------------------------------------------------------------------
# the same in plain float64 torch
# ---------------------------------------------------------------------------------------------
class _Method:
    """The discrete method on a periodic box (face i - 1/2 along d is stored at index i)."""

    def __init__(self, p, n, tol):
        self.p, self.dim, self.n, self.tol = p, p["dim"], n, tol
        self.h = p["L"] / n[0]

    def S(self, a, d, k):
        return torch.roll(a, -k, self.dim - 1 - d)

    def D(self, u):
        return sum((self.S(v, d, 1) - v) / self.h for d, v in enumerate(u))

    def G(self, q):
        return [(q - self.S(q, d, -1)) / self.h for d in range(self.dim)]

    def avg(self, q, d):
        return 0.5 * (q + self.S(q, d, -1))

    def central(self, q):
        return [(self.S(q, d, 1) - self.S(q, d, -1)) / (2.0 * self.h) for d in range(self.dim)]

    def lap(self, q):
        return sum(self.S(q, d, 1) - 2.0 * q + self.S(q, d, -1)
                   for d in range(self.dim)) / self.h ** 2

    def mix(self, phi, a, b):
        # (the slope is zero where the clip is active, its ends included)
        return b + (a - b) * torch.where((phi > 0.0) & (phi < 1.0), phi,
                                         phi.detach().clamp(0.0, 1.0))

    def rho(self, phi):
        return self.mix(phi, self.p["rho_in"], self.p["rho_out"])

    def normals(self, q):
        g = self.central(q)
        mag2 = sum(v * v for v in g)
        mag = torch.where(mag2 > 0, torch.sqrt(torch.where(mag2 > 0, mag2, 1.0)), 0.0)
        return [v / (mag + self.p["delta_n"]) for v in g], mag

    def flux(self, phi, u, gamma, d, nrm, psi):
        pf, eps = self.avg(phi, d), self.p["eps"]
        if psi is None:
            sharp = pf * (1.0 - pf)
        else:
            sharp = 0.25 * (1.0 - torch.tanh(self.avg(psi, d) / (2.0 * eps)) ** 2)
        return u[d] * pf - gamma * (eps * (phi - self.S(phi, d, -1)) / self.h
                                    - sharp * self.avg(nrm[d], d))

    def rhs(self, phi, u, gamma):
        p, h, eps, sg = self.p, self.h, self.p["eps"], self.p["sigma"]
        dims = range(self.dim)
        psi = None
        if p["model"] == "acdi":
            q = phi.clamp(0.0, 1.0)
            psi = eps * torch.log((q + 1e-20) / (1.0 - q + 1e-20))
        nrm, mag = self.normals(phi if psi is None else psi)
        dwell = phi * (1.0 - phi) * (1.0 - 2.0 * phi)
        kap = None
        if p["model"] in ("sb", "isodi") or p["force"] != "eb":
            m = self.normals(phi)[0]
            kap = -sum((self.S(m[d], d, 1) - self.S(m[d], d, -1)) / (2.0 * h) for d in dims)
        if p["model"] in ("cdi", "acdi"):
            F = [self.flux(phi, u, gamma, d, nrm, psi) for d in dims]
            kphi = -self.D(F)
        else:
            third = eps * mag * kap if p["model"] == "sb" else phi * (1.0 - phi) * kap
            kphi = -self.D([u[d] * self.avg(phi, d) for d in dims]) + gamma * (
                eps * self.lap(phi) - dwell / eps + third)
        eta = self.mix(phi, p["mu_in"], p["mu_out"])
        rc = self.rho(phi)
        cons = p["momentum"] == "consistent"
        if cons:
            m = [p["rho_out"] * u[d] + (p["rho_in"] - p["rho_out"]) * F[d] for d in dims]
        if p["force"] == "eb":
            mu = (6.0 * sg / eps) * dwell - 6.0 * sg * eps * self.lap(phi)
        gphi = self.G(phi)
        ku = []
        for d in dims:
            ud, adv, visc = u[d], 0.0, 0.0
            for e in dims:
                if e == d:
                    if cons:
                        f = 0.25 * (m[d] + self.S(m[d], d, 1)) * (ud + self.S(ud, d, 1))
                        adv = adv + (f - self.S(f, d, -1)) / h
                    else:
                        adv = adv + ud * (self.S(ud, d, 1) - self.S(ud, d, -1)) / (2.0 * h)
                    tau = 2.0 * eta * (self.S(ud, d, 1) - ud) / h
                    visc = visc + (tau - self.S(tau, d, -1)) / h
                else:
                    if cons:
                        f = 0.25 * (m[e] + self.S(m[e], d, -1)) * (ud + self.S(ud, e, -1))
                        adv = adv + (self.S(f, e, 1) - f) / h
                    else:
                        w = u[e] + self.S(u[e], d, -1)
                        w = 0.25 * (w + self.S(w, e, 1))
                        adv = adv + w * (self.S(ud, e, 1) - self.S(ud, e, -1)) / (2.0 * h)
                    ee = eta + self.S(eta, d, -1)
                    ee = 0.25 * (ee + self.S(ee, e, -1))
                    tau = ee * ((ud - self.S(ud, e, -1)) + (u[e] - self.S(u[e], d, -1))) / h
                    visc = visc + (self.S(tau, e, 1) - tau) / h
            if p["force"] == "eb":
                f = self.avg(mu, d) * gphi[d]
            else:
                f = sg * self.avg(kap, d) * gphi[d]
                if p["force"] == "lcsf":
                    pf = self.avg(phi, d)
                    f = 6.0 * f * pf * (1.0 - pf)
            ku.append(-adv + visc + f if cons else -adv + (visc + f) / self.avg(rc, d))
        return kphi, ku

    def solve(self, beta, b, x0=None):
        """Zero-mean x of -D(beta G x) = b - mean b: conjugate gradients preconditioned by the
        constant-coefficient inverse, to `tol` of the right-hand side."""
        b = b - b.mean()
        lam = 0.0
        for d in range(self.dim):
            k = torch.arange(self.n[d], dtype=torch.float64, device=b.device)
            v = [1] * self.dim
            v[self.dim - 1 - d] = self.n[d]
            e = ((2.0 - 2.0 * torch.cos(2.0 * math.pi * k / self.n[d])) / self.h ** 2).reshape(v)
            lam = lam + (e[..., : self.n[0] // 2 + 1] if d == 0 else e)
        inv = torch.where(lam > 0, 1.0 / torch.where(lam > 0, lam, 1.0), 0.0)
        # scaled by sqrt of the local density: the preconditioner sees the jump
        w = 0.5 * sum(q + self.S(q, d, 1) for d, q in enumerate(beta)) / self.dim
        w = w ** -0.5

        def M(r):
            z = w * torch.fft.irfftn(torch.fft.rfftn(w * r) * inv, s=r.shape)
            return z - z.mean()

        def A(x):
            return -self.D([bt * q for bt, q in zip(beta, self.G(x))])

        x = torch.zeros_like(b) if x0 is None else x0
        r = b - A(x)
        z = M(r)
        pd, rz = z, (r * z).sum()
        top = self.tol * float(b.norm())
        for _ in range(3000):
            if float(r.norm()) <= top:
                break
            q = A(pd)
            al = rz / (pd * q).sum()
            x = x + al * pd
            r = r - al * q
            z = M(r)
            new = (r * z).sum()
            pd, rz = z + (new / rz) * pd, new
        return x - x.mean()

    def project(self, phi, us, tau, x0=None):
        rc = self.rho(phi)
        beta = [1.0 / self.avg(rc, d) for d in range(self.dim)]
        pr = _Solve.apply(self, x0, -self.D(us) / tau, *beta)
        return [v - tau * bt * q for v, bt, q in zip(us, beta, self.G(pr))], pr

    def step(self, phi, u, gamma, x0=None):
        p, dt, dims = self.p, self.p["dt"], range(self.dim)
        cons = p["momentum"] == "consistent"

        def dens(f):
            rc = self.rho(f)
            return [self.avg(rc, d) if cons else 1.0 for d in dims]

        mn = [a * v for a, v in zip(dens(phi), u)]
        if p["scheme"] == "fe":
            kp, ku = self.rhs(phi, u, gamma)
            phi1 = phi + dt * kp
            us = [(m + dt * k) / a for m, k, a in zip(mn, ku, dens(phi1))]
            u1, pr = self.project(phi1, us, dt, x0)
            return phi1, u1, pr
        ps, us, pr = phi, u, x0
        accp, accu = phi, mn
        for s, (wt, cn) in enumerate(zip((1 / 6, 1 / 3, 1 / 3, 1 / 6), (0.5, 0.5, 1.0, 1.0))):
            kp, ku = self.rhs(ps, us, gamma)
            accp = accp + wt * dt * kp
            accu = [a + wt * dt * k for a, k in zip(accu, ku)]
            ps = phi + cn * dt * kp if s < 3 else accp
            m = [a + cn * dt * k for a, k in zip(mn, ku)] if s < 3 else accu
            us, pr = self.project(ps, [v / a for v, a in zip(m, dens(ps))], cn * dt,
                                  None if pr is None else pr.detach())
        return ps, us, pr


class _Solve(torch.autograd.Function):
    """x(b, beta) of the pressure system and its transpose."""

    @staticmethod
    def forward(ctx, m, x0, b, *beta):
        x = m.solve(beta, b, x0)
        ctx.m = m
        ctx.save_for_backward(x, *beta)
        return x

    @staticmethod
    def backward(ctx, g):
        x, *beta = ctx.saved_tensors
        lam = ctx.m.solve(beta, g)
        return (None, None, lam) + tuple(-a * b for a, b in zip(ctx.m.G(lam), ctx.m.G(x)))


def _double_box(p, phi, u):
    """The walled box and its mirror image as one periodic box (free-slip walls)."""
    v = u[1]
    return (torch.cat([phi, phi.flip(0)]),
            [torch.cat([u[0], u[0].flip(0)]),
             torch.cat([v, torch.zeros_like(v[:1]), -v[1:].flip(0)])])


def _exact_steps(p, seed, steps):
    phi, u = _inputs(p, seed)
    n = list(p["n"])
    if p["wall_y"]:
        phi, u = _double_box(p, phi, u)
        n[1] *= 2
    m = _Method(p, n, 1e-13 if p["precision"] == "fp64" else 1e-11)
    pr = None
    for _ in range(steps):
        phi, u, pr = m.step(phi, u, _gamma(u), pr)
    if p["wall_y"]:
        ny = p["n"][1]
        phi, u, pr = phi[:ny], [v[:ny] for v in u], pr[:ny]
    pr = pr - pr.mean()
    return phi.reshape(-1), torch.stack([v.reshape(-1) for v in u]), pr.reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        got = [_exact_steps(p, seed * 1000 + i, case["steps"])
               for i, p in enumerate(_batch_params(case))]
        return [torch.cat([torch.cat([f, u.reshape(-1)]) for f, u, _ in got]),
                torch.cat([q for _, _, q in got])]
    p = _params(case)
    if kind == "step":
        return list(_exact_steps(p, seed, case["steps"]))
    phi, u = _inputs(p, seed)
    m = _Method(p, p["n"], 1e-13)
    if kind == "solve":
        rc = m.rho(phi)
        return m.solve([1.0 / m.avg(rc, d) for d in range(m.dim)],
                       _rhs_field(p, phi, u)).reshape(-1)
    if kind == "rhs":
        kphi, ku = m.rhs(phi, u, _gamma(u))
        return [kphi.reshape(-1), torch.stack(ku).reshape(-1)]
    names = ("sigma", "rho_in", "rho_out", "mu_in", "mu_out")
    theta = [torch.tensor(p[k], dtype=torch.float64, device="cuda", requires_grad=True)
             for k in names]
    m.p = dict(p, **dict(zip(names, theta)))
    phi, u = phi.requires_grad_(), [v.requires_grad_() for v in u]
    phi1, u1, _ = m.step(phi, u, p["gamma_fixed"])
    lam = _cotangent(p, seed).reshape(1 + p["dim"], -1)
    J = sum((a.reshape(-1) * b).sum() for a, b in zip([phi1] + u1, lam))
    g = torch.autograd.grad(J, [phi] + u + theta)
    return [torch.cat([v.reshape(-1) for v in g[: 1 + p["dim"]]]), torch.stack(g[1 + p["dim"]:])]
