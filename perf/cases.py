"""The work that users of this framework have it do, as cases to be timed.

A pass is one call of the public entry points on data that a user's program holds on
the GPU: time steps of one field (every precision, scheme, scattering kernel, radial
grid and form), a differentiated run (forward, recomputation and adjoint), and a batched
step of many uneven problems. Sizes are those of this repository's benchmark and tests
(17 x 8^4, 33 x 16^4, 65 x 32^4, the 129 x 16 x 16 x 24 x 16 Lambert shell, the uneven
batch) and ragged ones of the same range.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1104_5330_gb300.ts as ts
from paper_1104_5330_gb300 import autograd as tsgrad

R1, R2 = 0.2, 1.0
PRECISION = {"f64": ts.TS_FP64, "f32": ts.TS_FP32, "f32r64": ts.TS_FP32_R64,
             "tf32x3": ts.TS_TF32X3, "bf16x3": ts.TS_BF16X3}
SCHEME = {"rk4": ts.TS_RK4, "split": ts.TS_RK4_SPLIT_IMPLICIT, "ab2": ts.TS_AB2}
RADIAL = {"cheb": ts.TS_RADIAL_CHEBYSHEV, "fd": ts.TS_RADIAL_UPWIND_FD,
          "zoned": ts.TS_RADIAL_ZONED}
FORM = {"plain": ts.TS_FORM_ADVECTIVE, "cons": ts.TS_FORM_CONSERVATIVE}


def _step(Nr, Nt, Np, NT, NP, groups, precision="f64", scheme="rk4", scatter="iso",
          radial="cheb", form="plain", zone=0, steps=1, moments=False, **more):
    return dict(kind="step", Nr=Nr, Nt=Nt, Np=Np, NT=NT, NP=NP, groups=groups,
                precision=precision, scheme=scheme, scatter=scatter, radial=radial, form=form,
                zone=zone, steps=steps, moments=moments, **more)


def listed():
    return [
        # a single small problem, as in a parameter study or an interactive run: latency counts
        _step(17, 8, 8, 8, 8, 1, name="small_f64"),
        # the benchmark's workload: absorber, four energy groups, double precision
        _step(33, 16, 16, 16, 16, 4, name="absorber_f64"),
        # the same in single precision
        _step(33, 16, 16, 16, 16, 4, "f32", name="absorber_f32"),
        # and with the radial contraction in split TF32
        _step(33, 16, 16, 16, 16, 4, "tf32x3", name="absorber_tf32x3"),
        # one finely resolved group, the largest field of the benchmark
        _step(65, 32, 32, 32, 32, 1, name="fine_f64"),
        # the precision workload at that size: single precision, double radial end rows
        _step(65, 32, 32, 32, 32, 1, "f32r64", name="fine_f32r64"),
        # the paper's own time marching with Thomson scattering, two steps a call
        _step(33, 16, 16, 16, 16, 4, scheme="ab2", scatter="thomson", steps=2,
              name="thomson_ab2_f64"),
        # the Lambert-shell run on the hybrid radial grid, with the moments a run looks at
        _step(129, 16, 16, 24, 16, 1, scatter="shell", radial="fd", moments=True,
              name="lambert_shell_f64"),
        # ragged sizes with the neutrino-nucleon kernel and the implicit collision step
        _step(21, 12, 10, 14, 12, 6, scheme="split", scatter="linear", name="ragged_split_f64"),
        # the conservative form of the benchmark's workload
        _step(33, 16, 16, 16, 16, 4, form="cons", name="conservative_f64"),
        # sensitivities of the outgoing flux: four steps, their recomputation and the adjoint
        dict(kind="gradient", Nr=33, Nt=16, Np=16, NT=16, NP=16, groups=8, precision="f64",
             scheme="rk4", steps=4, name="gradient_f64"),
        # many uneven problems stepped together, as in the batch benchmark
        dict(kind="batch", n=16, max_groups=6, mix=1104, precision="f32r64", scheme="split",
             name="batch_f32r64"),
    ]


_MOST = 12_000_000     # points of a drawn field: the slowest forms stay below the largest listed case


def draw(rng):
    def log_int(lo, hi, unit=1):
        v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(lo, v // unit * unit)

    def sizes():
        if rng.random() < 0.4:
            n = rng.choice([8, 16, 24, 32])
            return n, n, n, n
        return log_int(4, 32), log_int(4, 32, 2), log_int(4, 32, 2), log_int(8, 32, 4)

    what = rng.random()
    if what < 0.12:
        return dict(kind="batch", n=rng.randint(3, 12), max_groups=rng.randint(1, 4),
                    mix=rng.randrange(1 << 20), precision=rng.choice(["f32r64", "f32", "f64"]),
                    scheme=rng.choice(["split", "rk4", "ab2"]))
    while True:
        Nt, Np, NT, NP = sizes()
        if rng.random() < 0.3:
            Nr = rng.choice([17, 33, 65])
        else:
            Nr = log_int(9, 97)
        S = Nr * Nt * Np * NT * NP
        if S > _MOST:
            continue
        groups = min(log_int(1, 24), max(1, _MOST // S))
        break
    if what < 0.27:
        return dict(kind="gradient", Nr=Nr, Nt=Nt, Np=Np, NT=NT, NP=NP,
                    groups=max(1, min(groups, 3_000_000 // S)),
                    precision="f64", scheme=rng.choice(["rk4", "rk4", "ab2"]),
                    steps=rng.randint(1, 4))
    radial = rng.choice(["cheb"] * 5 + ["fd", "zoned"])
    form = "cons" if radial == "cheb" and rng.random() < 0.15 else "plain"
    precision = rng.choice(["f64", "f32"] if radial != "cheb" else
                           ["f64", "f64", "f64", "f32", "f32", "f32r64", "tf32x3", "bf16x3"])
    scheme = rng.choice(["rk4", "rk4", "ab2"] if form == "cons" else ["rk4", "rk4", "ab2", "split"])
    scatter = rng.choice(["iso", "iso", "linear", "thomson"]) if NT >= 6 else "iso"
    zone = 0
    if radial == "zoned":
        zone = rng.randint(4, 30)
        Nr = min(123, rng.randint(9, 65) + 2 * (zone - 1))
        groups = max(1, min(groups, _MOST // (Nr * Nt * Np * NT * NP)))
    return _step(Nr, Nt, Np, NT, NP, groups, precision, scheme, scatter, radial, form, zone,
                 rng.randint(1, 3), precision == "f64" and form == "plain" and rng.random() < 0.25)


# ------------------------------------------------------------------ inputs
def _zone_width(c):
    return 0.1


def _nodes(c):
    """Nodes of the five axes (float64 tensors on the host)."""
    Nr = c["Nr"]
    i = np.arange(Nr)
    radial = c.get("radial", "cheb")
    if radial == "fd":
        r = R1 + (R2 - R1) * i / (Nr - 1)
    elif radial == "zoned":
        nA = c["zone"]
        nB = Nr - 2 * (nA - 1)
        w = _zone_width(c) * (R2 - R1)
        e = w * np.arange(nA) / (nA - 1)
        mid = 0.5 * (R1 + R2) - (0.5 * (R2 - R1) - w) * np.cos(np.pi * np.arange(nB) / (nB - 1))
        r = np.concatenate([R1 + e, mid[1:-1], R2 - w + e])
    else:
        r = 0.5 * (R1 + R2) - 0.5 * (R2 - R1) * np.cos(np.pi * i / (Nr - 1))
    half = lambda n: np.pi * (np.arange(n) + 0.5) / n
    full = lambda n: 2 * np.pi * np.arange(n) / n
    return [torch.from_numpy(np.ascontiguousarray(x)) for x in
            (r, half(c["Nt"]), full(c["Np"]), half(c["NT"]), full(c["NP"]))]


def _time_step(c):
    """A stable step: the radial Courant limit, and the angular ones where they are smaller."""
    r, th, _, _, _ = _nodes(c)
    h = float((r[1:] - r[:-1]).min())
    t0 = float(th[0])
    angular = (c["Nt"] / 2 + c["Np"] / 2 / math.sin(t0) + c["NT"] / 2
               + c["NP"] / 2 / math.tan(t0)) / R1
    dt = min(0.4 * h, 1.2 / angular)
    return 0.4 * dt if c["scheme"] == "ab2" else dt


def _shape(c):
    return (c["groups"], c["Nr"], c["Nt"], c["Np"], c["NT"], c["NP"])


def _smooth(c, gen, dev):
    """A smooth distribution per group: a random polynomial of the position's unit
    vector, the direction and the Chebyshev variable of r (float64)."""
    r, th, ph, Th, Ph = (x.to(dev) for x in _nodes(c))
    sth, cth = torch.sin(th)[:, None], torch.cos(th)[:, None]
    sph, cph = torch.sin(ph)[None], torch.cos(ph)[None]
    one = torch.ones_like(sph)
    pos = [sth * cph, sth * sph, cth * one]                       # e_r
    eth = [cth * cph, cth * sph, -sth * one]
    eph = [-sph + 0 * sth, cph + 0 * sth, 0 * (sth * one)]
    a, b, d = (torch.cos(Th)[:, None] * torch.ones_like(Ph)[None],
               torch.sin(Th)[:, None] * torch.cos(Ph)[None],
               torch.sin(Th)[:, None] * torch.sin(Ph)[None])
    om = [p[:, :, None, None] * a + e[:, :, None, None] * b + f[:, :, None, None] * d
          for p, e, f in zip(pos, eth, eph)]
    x = ((2 * r - R1 - R2) / (R2 - R1)).clamp(-1, 1)
    F = torch.empty(_shape(c), dtype=torch.float64, device=dev)
    for g in range(c["groups"]):
        w = torch.randn(4, 10, generator=gen, dtype=torch.float64).to(dev)
        ang = []
        for k in range(4):
            u = [w[k, 0] + sum(w[k, 1 + q] * pos[q] for q in range(3))]
            q = u[0][:, :, None, None] + sum(w[k, 4 + q] * om[q] for q in range(3))
            q = q + 0.5 * (w[k, 7] * om[0] * om[1] + w[k, 8] * om[2] ** 2
                           + w[k, 9] * pos[0][:, :, None, None] * om[2])
            ang.append(q * 2.0 ** -k)
        cheb = [torch.ones_like(x), x, 2 * x * x - 1, 4 * x ** 3 - 3 * x]
        F[g] = 2.0
        for k in range(4):
            F[g] += 0.25 * cheb[k][:, None, None, None, None] * ang[k][None]
    return F


def _coefficients(c, gen, dev):
    """kappa, eta, kappa_s and the kernel's b, c on [G][Nr][Nt][Np] (float64)."""
    r, th, ph, _, _ = (x.to(dev) for x in _nodes(c))
    G = c["groups"]
    amp = (0.8 + 0.4 * torch.rand(G, 4, generator=gen, dtype=torch.float64)).to(dev)
    u = (torch.sin(th)[:, None] * torch.cos(ph)[None])[None, None]
    rr = r[None, :, None, None]
    s = lambda q: amp[:, q][:, None, None, None]
    if c.get("scatter") == "shell":      # scattering plasma of optical depth 5, densest inside
        ks = s(0) * 45.0 / (R2 - R1) * (1 + 0.1 * rr * u) * (1 - (rr - R1) / (R2 - R1)) ** 8
        return torch.zeros_like(ks), torch.zeros_like(ks), ks.contiguous(), None, None
    scale = c.get("kappa_scale", 1.0)
    kap = scale * s(0) * (1 + 0.5 * u + 0 * rr)
    eta = kap * torch.exp(-s(1) * rr ** 2)
    ks = 0.5 * s(2) * torch.ones_like(kap)
    b = cq = None
    if c.get("scatter") == "linear":     # neutrinos on a neutron/proton mixture
        b = -(0.25 + 0.08 * s(3) * u * torch.ones_like(rr)).contiguous()
    elif c.get("scatter") == "thomson":
        cq = torch.full_like(kap, 0.75)
    return kap.contiguous(), eta.contiguous(), ks.contiguous(), b, cq


def _jacobian(c, dev):
    r, th, _, Th, _ = (x.to(dev) for x in _nodes(c))
    return ((r ** 2)[:, None, None, None, None] * torch.sin(th)[:, None, None, None]
            * torch.sin(Th)[:, None])


def _inputs(c, seed, dev):
    """What defines one problem: fields, coefficients, inflow data and the step."""
    gen = torch.Generator().manual_seed(1_000_003 * int(seed) + 17)
    double = c["precision"] == "f64"
    h = c["NT"] // 2
    coef = _coefficients(c, gen, dev)
    if c.get("scatter") == "shell":      # an empty shell lit by a Lambert emitter at R1
        Th = _nodes(c)[3].to(dev)
        F = torch.zeros(_shape(c), dtype=torch.float64, device=dev)
        amp = 1 + torch.rand(c["groups"], generator=gen, dtype=torch.float64).to(dev)
        F[:, 0, :, :, :h] = amp[:, None, None, None, None] * torch.cos(Th[:h])[:, None]
    else:
        F = _smooth(c, gen, dev)
        if c.get("form") == "cons":
            F *= _jacobian(c, dev)
    if not double:
        F = F.float()
    return F, coef, F[:, 0, :, :, :h].clone(), F[:, -1, :, :, h:].clone()


def _batch_problems(c):
    rng = random.Random(c["mix"])
    out = []
    for _ in range(c["n"]):
        Nt, Np, NT, NP = (rng.choice([8, 16, 24]) for _ in range(4))
        out.append(dict(Nr=rng.choice([17, 33, 65]), Nt=Nt, Np=Np, NT=NT, NP=NP,
                        groups=rng.randint(1, c["max_groups"]), precision=c["precision"],
                        scheme=c["scheme"], scatter="iso", radial="cheb", form="plain",
                        kappa_scale=math.exp(rng.uniform(math.log(0.1), math.log(100.0)))
                        if c["scheme"] == "split" else rng.uniform(0.1, 5.0)))
    return out


def _desc(c):
    return ts.GridDesc(R1, R2, c["Nr"], c["Nt"], c["Np"], c["NT"], c["NP"], c["groups"],
                       PRECISION[c["precision"]], SCHEME[c["scheme"]], ts.TS_BC_TAU_INFLOW, 0,
                       36.0, 16, 0, 0, 0.0, 0)


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "batch":
        problems = _batch_problems(case)
        batch = ts.Batch([_desc(p) for p in problems])
        fields = []
        for q, (p, g) in enumerate(zip(problems, batch.grids)):
            F, (kap, eta, ks, _, _), g1, g2 = _inputs(p, 97 * seed + q, dev)
            g.set_coeffs(kap, eta, ks, g1, g2)
            fields.append(F)
        return dict(kind="batch", batch=batch, fields=fields,
                    dts=[_time_step(p) for p in problems])
    F, (kap, eta, ks, b, cq), g1, g2 = _inputs(case, seed, dev)
    grid = ts.Grid(R1, R2, case["Nr"], case["Nt"], case["Np"], case["NT"], case["NP"],
                   case["groups"], precision=PRECISION[case["precision"]],
                   scheme=SCHEME[case["scheme"]], radial=RADIAL[case.get("radial", "cheb")],
                   zone_nodes=case.get("zone", 0),
                   zone_width=_zone_width(case) if case.get("zone", 0) else 0.0,
                   form=FORM[case.get("form", "plain")])
    state = dict(kind=case["kind"], grid=grid, F=F, dt=_time_step(case), steps=case["steps"])
    if case["kind"] == "gradient":
        state.update(kappa=kap.requires_grad_(), eta=eta.requires_grad_(), kappa_s=ks,
                     F=F.requires_grad_(), inflow=(g1, g2))
        return state
    grid.set_coeffs(kap, eta, ks, g1, g2)
    if b is not None:
        grid.set_scattering_anisotropy(b)
    if cq is not None:
        grid.set_scattering_quadrupole(cq)
    state["moments"] = case["moments"]
    return state


def run(state):
    if state["kind"] == "batch":
        return state["batch"].step(state["fields"], state["dts"])
    grid = state["grid"]
    if state["kind"] == "gradient":
        F0, kappa, eta = state["F"], state["kappa"], state["eta"]
        F = tsgrad.transport_steps(grid, F0, kappa, eta, state["kappa_s"], state["dt"],
                                   state["steps"], *state["inflow"])
        J = tsgrad.outgoing_flux(grid, F)
        gF, gk, ge = torch.autograd.grad(J.sum(), [F0, kappa, eta])
        return dict(F=F.detach(), J=J.detach(), gF=gF, gkappa=gk, geta=ge)
    F = grid.step(state["F"], state["dt"], state["steps"])
    if state["moments"]:
        return (F,) + grid.moments(F)
    return F


def _one_work(c):
    pts = math.prod(_shape(c))
    es = 8 if c["precision"] == "f64" else 4
    coef = 8 * math.prod(_shape(c)[:4])
    # one stage derivative: the per-axis contractions in their folded forms, and the
    # pointwise work of the operator and of the stage update
    radial = 4 if c.get("radial", "cheb") == "fd" else c["Nr"] + 1
    flops = c["Nt"] + c["Np"] + c["NT"] + c["NP"] + radial + 45
    stages = 1 if c["scheme"] == "ab2" else 4
    n = c.get("steps", 1)
    # a step reads and writes the field (AB2 also its kept derivative)
    per_step = (4 if c["scheme"] == "ab2" else 2) * es * pts + 3 * coef
    return n * per_step, n * stages * flops * pts


def work(case):
    if case["kind"] == "batch":
        both = [_one_work(p) for p in _batch_problems(case)]
        return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}
    nbytes, flops = _one_work(case)
    if case["kind"] == "gradient":   # forward, recomputation, and the transposed operator
        return {"bytes": 3 * nbytes, "flops": 3 * flops}
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ in 64 bits
def _fourier(M):
    j = torch.arange(M, dtype=torch.float64)
    q = j[:, None] - j[None, :]
    t = torch.tan(q * math.pi / M)
    sign = 1 - 2 * (q.abs() % 2)
    D = 0.5 * sign / torch.where(q == 0, torch.ones_like(t), t)
    if M % 2 == 0:   # cot(pi/2) is zero
        D[(q.abs() * 2 == M)] = 0.0
    return D.masked_fill(q == 0, 0.0)


def _chebyshev(n, a, b):
    """D on the n Gauss-Lobatto nodes of [a, b], ascending."""
    N = n - 1
    i = torch.arange(n, dtype=torch.float64)
    cb = torch.ones(n, dtype=torch.float64)
    cb[0] = cb[-1] = 2.0
    cb = cb * (1 - 2 * (i % 2))
    dx = (2 * torch.sin(math.pi * (i[:, None] + i[None, :]) / (2 * N))
          * torch.sin(math.pi * (i[:, None] - i[None, :]) / (2 * N)))
    D = cb[:, None] / cb[None, :] / torch.where(dx == 0, torch.ones_like(dx), dx)
    D.fill_diagonal_(0.0)
    D -= torch.diag(D.sum(1))
    return D * 2 / (b - a)


def _fejer(N):
    t = math.pi * (torch.arange(N, dtype=torch.float64) + 0.5) / N
    m = torch.arange(1, N // 2 + 1, dtype=torch.float64)
    return 2 / N * (1 - 2 * (torch.cos(2 * m[None] * t[:, None]) / (4 * m * m - 1)[None]).sum(1))


def _clenshaw_curtis(n):
    N = n - 1
    i = torch.arange(n, dtype=torch.float64)
    k = torch.arange(1, N // 2 + 1, dtype=torch.float64)
    b = torch.where(2 * k == N, 1.0, 2.0)
    w = 1 - ((b / (4 * k * k - 1))[None] * torch.cos(2 * k[None] * i[:, None] * math.pi / N)).sum(1)
    w = w * 2 / N
    w[0] /= 2
    w[-1] /= 2
    return w


def _along(M, F, axis):
    """M applied along one axis of F."""
    s = F.shape
    left, right = math.prod(s[:axis]), math.prod(s[axis + 1:])
    if right == 1:
        return (F.reshape(left, s[axis]) @ M.T).reshape(s)
    return torch.matmul(M, F.reshape(left, s[axis], right)).reshape(s)


class _Operator:
    """dF/dt of one problem and its time stepping, dense and in 64 bits."""

    def __init__(self, c, coef, dev):
        self.c, self.coef = c, list(coef)
        r, th, ph, Th, Ph = (x.to(dev) for x in _nodes(c))
        v = lambda x, ax: x.reshape([-1 if a == ax else 1 for a in range(6)])
        self.r, self.th, self.Th, self.Ph = v(r, 1), v(th, 2), v(Th, 4), v(Ph, 5)
        sg = -1.0 if c.get("form") == "cons" else 1.0
        n = lambda M: M.to(dev).contiguous()

        def doubled(N):
            D = _fourier(2 * N)
            return n(D[:N, :N]), n(sg * D[:N, N:].flip(1))

        self.At, self.Bt = doubled(c["Nt"])
        self.AT, self.BT = doubled(c["NT"])
        self.Dp, self.DP = n(_fourier(c["Np"])), n(_fourier(c["NP"]))
        self.q = (_fejer(c["NT"]) / (2 * c["NP"])).to(dev).reshape(1, 1, 1, 1, -1, 1)
        self.out = torch.cos(self.Th) > 0
        self.radial = c.get("radial", "cheb")
        Nr = c["Nr"]
        if self.radial == "cheb":
            self.Dr = n(_chebyshev(Nr, R1, R2))
            i = torch.arange(Nr, dtype=torch.float64, device=dev)
            self.tn = v(1 - 2 * ((Nr - 1 - i) % 2), 1)
        elif self.radial == "zoned":
            self.nA = c["zone"]
            self.nB = Nr - 2 * (self.nA - 1)
            w = _zone_width(c) * (R2 - R1)
            self.hA = w / (self.nA - 1)
            self.DB = n(_chebyshev(self.nB, R1 + w, R2 - w))
            i = torch.arange(self.nB, dtype=torch.float64, device=dev)
            self.tn = v(1 - 2 * ((self.nB - 1 - i) % 2), 1)
        J = _jacobian(c, dev) if c.get("form") == "cons" else None
        self.jac = None if J is None else J[None]
        if J is not None:   # the removal of the Nyquist bin of the doubled Theta circle
            N = c["NT"]
            alt = (1 - 2 * (torch.arange(2 * N, dtype=torch.float64) % 2)) / math.sqrt(2 * N)
            P = torch.eye(2 * N, dtype=torch.float64) - alt[:, None] * alt[None, :]
            self.PA, self.PB = n(P[:N, :N]), n(-P[:N, N:].flip(1))

    def halfturn(self, F, both):
        F = torch.roll(F, -(self.c["NP"] // 2), 5)
        return torch.roll(F, -(self.c["Np"] // 2), 3) if both else F

    def d_r(self, F):
        if self.radial == "cheb":
            return _along(self.Dr, F, 1)
        Nr = F.shape[1]
        if self.radial == "fd":
            h = (R2 - R1) / (Nr - 1)
            z = torch.zeros_like(F[:, :1])
            d = (F[:, 1:] - F[:, :-1]) / h
            return torch.where(self.out, torch.cat([z, d], 1), torch.cat([d, z], 1))
        a, b = self.nA - 1, self.nA - 1 + self.nB - 1
        z = torch.zeros_like(F[:, :1])
        d = (F[:, 1:] - F[:, :-1]) / self.hA
        back, fwd = torch.cat([z, d], 1), torch.cat([d, z], 1)
        dB = _along(self.DB, F[:, a:b + 1], 1)
        up = dB + (back[:, a:a + 1] - dB[:, :1]) * (self.tn / self.tn[:, :1])
        dn = dB + (fwd[:, b:b + 1] - dB[:, -1:]) * (self.tn / self.tn[:, -1:])
        up = torch.cat([back[:, :a + 1], up[:, 1:], back[:, b + 1:]], 1)
        dn = torch.cat([fwd[:, :a], dn[:, :-1], fwd[:, b:]], 1)
        return torch.where(self.out, up, dn)

    def streaming(self, F):
        sT, cT, cP, sP = torch.sin(self.Th), torch.cos(self.Th), torch.cos(self.Ph), torch.sin(self.Ph)
        sth, cth, r = torch.sin(self.th), torch.cos(self.th), self.r
        L = cT * self.d_r(F)
        L = L + sT * cP / r * (_along(self.At, F, 2) + _along(self.Bt, self.halfturn(F, True), 2))
        L = L + sT * sP / (r * sth) * _along(self.Dp, F, 3)
        H = self.halfturn(F, False)
        d = _along(self.AT, F, 4) + _along(self.BT, H, 4)
        if self.jac is None:
            return L - sT / r * d - sT * sP * cth / (r * sth) * _along(self.DP, F, 5)
        p = _along(self.PA, F, 4) + _along(self.PB, H, 4)
        return (L - (sT * d + cT * p) / r
                - sT * cth / (r * sth) * _along(self.DP, sP * F, 5))

    def mean(self, X):
        return (self.q * X).sum((4, 5), keepdim=True)

    def basis(self):
        sT, cT = torch.sin(self.Th), torch.cos(self.Th)
        cP, sP = torch.cos(self.Ph), torch.sin(self.Ph)
        return [cT * torch.ones_like(cP), sT * cP, sT * sP]

    def collision(self, F):
        kap, eta, ks, b, cq = (None if x is None else x[..., None, None] for x in self.coef)
        if self.jac is not None:
            F = F / self.jac
        J = self.mean(F)
        gain = J
        om = self.basis()
        if b is not None:
            gain = gain + b * sum(o * self.mean(o * F) for o in om)
        if cq is not None:
            gain = gain + cq * (sum(om[i] * om[j] * self.mean(om[i] * om[j] * F)
                                    for i in range(3) for j in range(3)) - J / 3)
        CT = eta - kap * F + ks * (gain - F)
        return CT if self.jac is None else self.jac * CT

    def rhs(self, F, collide=True):
        K = -self.streaming(F)
        if collide:
            K = K + self.collision(F)
        if self.radial == "cheb":     # Tau: the top Chebyshev mode takes the inflow node's rate
            at0 = K[:, :1] * self.tn[:, :1]
            atN = K[:, -1:] * self.tn[:, -1:]
            return K - torch.where(self.out, at0, atN) * self.tn
        keep = torch.ones(1, F.shape[1], 1, 1, F.shape[4], 1, dtype=F.dtype, device=F.device)
        h = self.c["NT"] // 2
        keep[:, 0, :, :, :h] = 0.0
        keep[:, -1, :, :, h:] = 0.0
        return K * keep

    def implicit(self, F, dt, g1, g2):
        """Backward-Euler collision: per position the linear system of the moments."""
        kap, eta, ks, b, cq = (None if x is None else x[..., None, None] for x in self.coef)
        den = 1 + dt * (kap + ks)
        J0 = self.mean(F)
        Jn = (J0 + dt * eta) / (1 + dt * kap)
        om = self.basis()
        gain = Jn
        if b is not None:
            f = b / (1 + dt * (kap + ks) - dt * ks * b / 3)
            gain = gain + f * sum(o * self.mean(o * F) for o in om)
        if cq is not None:
            f = cq / (1 + dt * (kap + ks) - dt * ks * cq * (2.0 / 15.0))
            M = sum(om[i] * om[j] * self.mean(om[i] * om[j] * F) for i in range(3) for j in range(3))
            gain = gain + f * (M - J0 / 3)
        F = (F + dt * (eta + ks * gain)) / den
        h = self.c["NT"] // 2
        F[:, 0, :, :, :h] = g1
        F[:, -1, :, :, h:] = g2
        return F

    def steps(self, F, dt, n, g1, g2):
        scheme = self.c["scheme"]
        last = None
        for _ in range(n):
            if scheme == "ab2":
                K = self.rhs(F)
                F = F + dt * (K if last is None else 1.5 * K - 0.5 * last)
                last = K
                continue
            full = scheme != "split"
            k1 = self.rhs(F, full)
            k2 = self.rhs(F + 0.5 * dt * k1, full)
            k3 = self.rhs(F + 0.5 * dt * k2, full)
            k4 = self.rhs(F + dt * k3, full)
            F = F + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
            if not full:
                F = self.implicit(F, dt, g1, g2)
        return F

    def flux(self, F, i, R):
        wth = _fejer(self.c["Nt"]).to(F.device)[:, None]
        m = (self.q * torch.cos(self.Th) * F[:, i:i + 1]).sum((4, 5))[:, 0]
        return R * R * 4 * math.pi * (2 * math.pi / self.c["Np"]) * (wth * m).sum((1, 2))

    def moments(self, F):
        c, dev = self.c, F.device
        _, th, ph, _, _ = (x.to(dev) for x in _nodes(c))
        s, (m0, m1, m2) = self.mean(F)[..., 0, 0], (self.mean(o * F)[..., 0, 0] for o in self.basis())
        sth, cth, sph, cph = torch.sin(th)[:, None], torch.cos(th)[:, None], torch.sin(ph), torch.cos(ph)
        F1 = torch.stack([m0 * sth * cph + m1 * cth * cph - m2 * sph,
                          m0 * sth * sph + m1 * cth * sph + m2 * cph, m0 * cth - m1 * sth])
        if self.radial == "cheb":
            w = _clenshaw_curtis(c["Nr"]) * 0.5 * (R2 - R1)
        elif self.radial == "fd":
            w = torch.full((c["Nr"],), (R2 - R1) / (c["Nr"] - 1), dtype=torch.float64)
            w[0] /= 2
            w[-1] /= 2
        else:
            w = torch.zeros(c["Nr"], dtype=torch.float64)
            e = torch.full((self.nA,), self.hA, dtype=torch.float64)
            e[0] /= 2
            e[-1] /= 2
            w[:self.nA] += e
            w[-self.nA:] += e
            a = self.nA - 1
            w[a:a + self.nB] += _clenshaw_curtis(self.nB) * (0.5 * (R2 - R1) - _zone_width(c) * (R2 - R1))
        w = (w.to(dev) * self.r.reshape(-1) ** 2)[:, None, None]
        wth = _fejer(c["Nt"]).to(dev)[:, None]
        N = (w * wth * s).sum((1, 2, 3)) * 4 * math.pi * 2 * math.pi / c["Np"]
        return s, F1, N, self.flux(F, 0, R1), self.flux(F, c["Nr"] - 1, R2)


def exact(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "batch":
        if case["scheme"] == "split" and sum(math.prod(_shape(p)) for p in _batch_problems(case)) > 6e8:
            return None
        out = []
        for q, p in enumerate(_batch_problems(case)):
            F, coef, g1, g2 = _inputs(p, 97 * seed + q, dev)
            op = _Operator(p, coef, dev)
            out.append(op.steps(F.double(), _time_step(p), 1, g1.double(), g2.double()).cpu())
        return out
    F, coef, g1, g2 = _inputs(case, seed, dev)
    dt, n = _time_step(case), case["steps"]
    if case["kind"] == "gradient":
        F = F.double().requires_grad_()
        kap, eta = coef[0].requires_grad_(), coef[1].requires_grad_()
        op = _Operator(case, coef, dev)
        Fn = op.steps(F, dt, n, None, None)
        J = op.flux(Fn, case["Nr"] - 1, R2)
        gF, gk, ge = torch.autograd.grad(J.sum(), [F, kap, eta])
        return dict(F=Fn.detach(), J=J.detach(), gF=gF, gkappa=gk, geta=ge)
    op = _Operator(case, coef, dev)
    Fn = op.steps(F.double(), dt, n, g1.double(), g2.double())
    return (Fn,) + op.moments(Fn) if case["moments"] else Fn
