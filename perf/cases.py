"""Performance cases of the relativistic lattice Boltzmann framework.

Each case is one piece of work a user's program asks for through the public entry
points (Lattice, TubeBatch, misfit_gradient, shock_tube_misfit) with the inputs in hand
on the GPU:

  run     a lattice is set to the equilibrium of given fields, advanced by `steps` time
          steps and its macroscopic fields are read back (with the conserved totals
          and the raw state where the program monitors or checkpoints the run);
  sweep   a batch of uneven shock tubes with its own relaxation times per tube, all
          advanced by `steps`;
  grad    the gradient of a profile misfit with respect to the relaxation times and the
          initial energy field, on a lattice the program keeps;
  fit     the same through the autograd function, as one iteration of a fit whose
          relaxation times change from call to call.

exact() states the scheme in plain torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1211_3286_gb300 import inputs as I
from paper_1211_3286_gb300.adjoint import misfit_gradient, shock_tube_misfit
from paper_1211_3286_gb300.batch import TubeBatch
from paper_1211_3286_gb300.lattice import Lattice

PER, ZG = "periodic", "zero_gradient"
DEV = "cuda"
FIELDS = ("e", "P", "ux", "uy", "uz", "n")
L2_BYTES = 129e6   # a state whose two copies exceed this has to pass through memory at every step


def _run(name=None, nx=1, ny=1, nz=1, steps=1, lattice="d3q19", precision="fp64", collision="mrt", tau_f=0.9, tau_v=0.9,
         tau_e=0.55, tau_eps=0.8, tau_q=0.0, bcx=PER, bcy=PER, bcz=PER, correction="", eta=0.0, umax=0.3,
         totals=False, state=False):
    c = dict(kind="run", nx=nx, ny=ny, nz=nz, steps=steps, lattice=lattice, precision=precision, collision=collision,
             tau_f=tau_f, tau_v=tau_v, tau_e=tau_e, tau_eps=tau_eps, tau_q=tau_q, bcx=bcx, bcy=bcy, bcz=bcz,
             correction=correction, eta=eta, umax=umax, totals=totals, state=state)
    return dict(c, name=name) if name else c


def _sweep(name=None, tubes=16, steps=400, precision="fp32", tuned=True):
    c = dict(kind="sweep", tubes=tubes, steps=steps, precision=precision, tuned=tuned)
    return dict(c, name=name) if name else c


def _grad(name=None, kind="grad", nx=1600, steps=400, collision="mrt"):
    c = dict(kind=kind, nx=nx, steps=steps, collision=collision, tau_v=0.9, tau_e=0.55, tau_eps=0.8)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a shock tube watched as it develops: a few steps between two looks at the fields
        # and the conserved totals (the smallest calls, bound by launches and latency)
        _run("tube_monitor", nx=1600, steps=20, bcx=ZG, totals=True),
        # the plain method's quasi-1D shock tube (Sec. III.B): single relaxation time
        _run("tube_bgk", nx=400, steps=2000, collision="bgk", tau_e=0.9, tau_eps=0.9, bcx=ZG),
        # the 3-D MRT box in FP64, the headline workload
        _run("box_fp64", nx=256, ny=256, nz=256, steps=20),
        # the same box at 512^3 with populations stored in FP32 (the largest case)
        _run("box_fp32_512", nx=512, ny=512, nz=512, steps=10, precision="fp32"),
        # a ragged box with open ends and its own energy-flux time, checkpointed at the end
        _run("box_ragged", nx=150, ny=110, nz=90, steps=40, tau_q=0.7, bcx=ZG, bcy=ZG, state=True),
        # the precision study's small box with FP32 storage
        _run("box_fp32_64", nx=64, ny=64, nz=64, steps=200, precision="fp32"),
        # fixed eta/s: relaxation times per node (Sec. III.B) on a box
        _run("box_eta", nx=128, ny=96, nz=80, steps=20, collision="mrt", tau_f=0.6, tau_e=0.05, tau_eps=0.05,
             tau_q=0.5, eta=0.02, umax=0.15),
        # the paper's D2Q9 MRT model with the C_7 correction on a plane
        _run("plane_c7", nx=1200, ny=900, steps=40, lattice="d2q9", tau_v=1.2, tau_f=1.2, tau_e=0.6, tau_eps=0.6,
             bcx=ZG, correction="c7", umax=0.2),
        # the discontinuity study: 1024 uneven tubes, launch shape tuned once
        _sweep("sweep_1024", tubes=1024, steps=400),
        # a handful of its tubes again in FP64, as a check, at the default launch shape
        _sweep("sweep_16_fp64", tubes=16, steps=400, precision="fp64", tuned=False),
        # the gradient through 4000 steps of a 1600-node tube
        _grad("grad_tube", nx=1600, steps=4000),
        # one iteration of a fit of the relaxation times and the initial field
        _grad("fit_tube", kind="fit", nx=800, steps=400),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "tube", "box", "box", "box", "plane", "plane", "sweep", "sweep", "grad", "fit"])
    taus = dict(tau_f=round(rng.uniform(0.6, 1.4), 3), tau_v=round(rng.uniform(0.7, 1.3), 3),
                tau_e=round(rng.uniform(0.55, 0.7), 3), tau_eps=round(rng.uniform(0.6, 0.9), 3))
    if kind == "tube":
        eta = rng.choice([0.0, 0.0, 0.0, 0.1])
        if eta:   # the Fig. 1 cases: BGK with tau_g per node, tau_f tied to it
            return _run(nx=_log(rng, 64, 6400), steps=_log(rng, 10, 2000), collision="bgk", tau_f=0.0, bcx=ZG, eta=eta)
        return _run(nx=_log(rng, 64, 6400), steps=_log(rng, 10, 2000), collision=rng.choice(["mrt", "bgk"]), bcx=ZG,
                    precision=rng.choice(["fp64", "fp64", "fp32"]), totals=rng.random() < 0.5, **taus)
    if kind == "box":
        nx, ny, nz = (_log(rng, 16, 240) for _ in range(3))
        most = max(4, int(3.0e8 / (nx * ny * nz)))
        bc = [rng.choice([PER, PER, PER, ZG]) for _ in range(3)]
        if rng.random() < 0.15:
            return _run(nx=nx, ny=ny, nz=nz, steps=min(most // 4 + 1, rng.randint(5, 40)), tau_f=0.6, tau_e=0.05,
                        tau_eps=0.05, tau_q=0.5, eta=0.02, umax=0.15, bcx=bc[0])
        return _run(nx=nx, ny=ny, nz=nz, steps=min(most, rng.randint(5, 60)), precision=rng.choice(["fp64", "fp32"]),
                    tau_q=rng.choice([0.0, 0.0, 0.0, 0.75]), bcx=bc[0], bcy=bc[1], bcz=bc[2],
                    totals=rng.random() < 0.5, **taus)
    if kind == "plane":
        te = round(rng.uniform(0.56, 0.7), 3)
        bc = [rng.choice([PER, ZG]) for _ in range(2)]
        return _run(nx=_log(rng, 40, 1600), ny=_log(rng, 40, 1600), steps=rng.randint(5, 60), lattice="d2q9",
                    tau_v=1.2, tau_f=round(rng.uniform(0.8, 1.4), 3), tau_e=te, tau_eps=te, bcx=bc[0], bcy=bc[1],
                    correction=rng.choice(["", "", "c7", "c7_printed"]), umax=0.2)
    if kind == "sweep":
        return _sweep(tubes=_log(rng, 6, 1024), steps=rng.randint(50, 400), precision=rng.choice(["fp32", "fp32", "fp64"]),
                      tuned=rng.random() < 0.5)
    return _grad(kind=kind, nx=_log(rng, 100, 1600), steps=_log(rng, 50, 2000 if kind == "grad" else 500),
                 collision=rng.choice(["mrt", "mrt", "bgk"]))


# ----------------------------------------------------------------------------- inputs
def _fields(c, seed):
    """Initial e, ux, uy, uz, n of a case on the GPU."""
    nx, ny, nz = c["nx"], c.get("ny", 1), c.get("nz", 1)
    if ny == 1 and nz == 1:
        state = I.PAPER_LATTICE_UNITS if c.get("eta", 0.0) else {}
        e, ux, uy, uz, n = (torch.from_numpy(a).to(DEV) for a in I.shock_tube(nx, **state))
        noise = torch.from_numpy(I.perturbation(2 * nx, seed=seed)).reshape(2, 1, 1, nx).to(DEV)
        return e * (1 + 1e-3 * noise[0]), ux, uy, uz, n * (1 + 1e-3 * noise[1])
    e0, n0 = (3 * 2.0e-7, 2.0e-7 / 0.0314) if c["eta"] else (1e-2, 1.0)
    e, ux, uy, uz, n = I.periodic_box(None, seed=seed, shape=(nz, ny, nx), device=DEV, umax=c["umax"], e0=e0, n0=n0)
    return [e, ux, uy, torch.zeros_like(uz) if c["lattice"] == "d2q9" else uz, n]


def _sweep_inputs(c, seed):
    lengths, taus = I.tube_sweep(c["tubes"])[0], I.tube_sweep(c["tubes"], seed=seed)[1]
    parts = [I.shock_tube(int(L)) for L in lengths]
    e, ux, uy, uz, n = (torch.from_numpy(np.concatenate([p[k].reshape(-1) for p in parts])).to(DEV) for k in range(5))
    noise = torch.from_numpy(I.perturbation(2 * e.numel(), seed=seed)).reshape(2, -1).to(DEV)
    return lengths, taus, [e * (1 + 1e-3 * noise[0]), ux, uy, uz, n * (1 + 1e-3 * noise[1])]


def _targets(c, seed):
    """Profiles to fit: a smoothed pressure step and a velocity plateau, with noise."""
    L, T = c["nx"], c["steps"]
    x = (torch.arange(L, dtype=torch.float64, device=DEV) - L / 2).reshape(1, 1, L)
    noise = torch.from_numpy(I.perturbation(L, seed=seed + 1)).reshape(1, 1, L).to(DEV)
    P = (2.22e-3 + (5.43e-3 - 2.22e-3) * 0.5 * (1 - torch.tanh(x / (0.3 * T + 8)))) * (1 + 1e-3 * noise)
    ux = 0.19 * torch.exp(-((x / (0.5 * T + 8)) ** 2))
    return [P, ux, torch.zeros_like(ux), torch.zeros_like(ux)]


def _lattice(c):
    return Lattice((c["nz"], c["ny"], c["nx"]), collision=c["collision"], tau_f=c["tau_f"], tau_v=c["tau_v"],
                   tau_e=c["tau_e"], tau_eps=c["tau_eps"], tau_q=c["tau_q"], bc=(c["bcx"], c["bcy"], c["bcz"]),
                   precision=c["precision"], lattice=c["lattice"], correction=c["correction"] or False,
                   eta_over_s=c["eta"])


def prepare(case, seed):
    c = dict(case, seed=seed)
    if c["kind"] == "run":
        return dict(c, fields=_fields(c, seed), lat=_lattice(c))
    if c["kind"] == "sweep":
        lengths, taus, fields = _sweep_inputs(c, seed)
        b = TubeBatch(lengths, taus, collision="mrt", precision=c["precision"])
        if c["tuned"]:
            b.set_fields(*fields)
            b.autotune(16)
        return dict(c, fields=fields, batch=b)
    s = dict(c, fields=_fields(c, seed), targets=_targets(c, seed))
    if c["kind"] == "grad":
        s["lat"] = Lattice((1, 1, c["nx"]), collision=c["collision"], tau_f=c["tau_v"], tau_v=c["tau_v"],
                           tau_e=c["tau_e"], tau_eps=c["tau_eps"], bc=(ZG, PER, PER))
    else:
        s["taus"] = [torch.tensor(c[k], dtype=torch.float64, device=DEV) for k in ("tau_v", "tau_e", "tau_eps")]
    return s


# ----------------------------------------------------------------------------- the work
def run(state):
    s = state
    if s["kind"] == "run":
        lat = s["lat"]
        lat.set_fields(*s["fields"])
        lat.step(s["steps"])
        out = dict(lat.fields())
        if s["totals"]:   # N0 and T00; the momenta of a periodic box are sums that cancel
            out["totals"] = lat.totals()[:2]
        if s["state"]:
            out["state"] = lat.state()
        return out
    if s["kind"] == "sweep":
        b = s["batch"]
        b.set_fields(*s["fields"])
        b.run(s["steps"])
        return b.fields()
    if s["kind"] == "grad":
        s["lat"].set_fields(*s["fields"])
        loss, dtau, de0 = misfit_gradient(s["lat"], s["steps"], *s["targets"])
        return {"loss": loss, "dtau": dtau, "de0": de0}
    e, ux, uy, uz, n = s["fields"]
    taus = [t.detach().requires_grad_(True) for t in s["taus"]]
    e0 = e.detach().requires_grad_(True)
    loss = shock_tube_misfit(*taus, e0, (ux, uy, uz), n, s["targets"], s["steps"], collision=s["collision"])
    loss.backward()
    return {"loss": loss.detach(), "dtau": torch.stack([t.grad for t in taus]), "de0": e0.grad}


def work(case):
    """Fields in and out once; a state too large for the chip's caches read and written at
    every step.  Flops of the scheme as written per node and step (D3Q19 440, D2Q9 200)."""
    c = case
    if c["kind"] == "run":
        q, size = (9, 8) if c["lattice"] == "d2q9" else (19, 8 if c["precision"] == "fp64" else 4)
        nodes = c["nx"] * c["ny"] * c["nz"]
        state = 2.0 * q * size * nodes
        b = (5 + 6) * 8.0 * nodes + (2.0 * state * c["steps"] if 2 * state > L2_BYTES else 0.0)
        return {"bytes": b + (state if c["state"] else 0.0), "flops": (440.0 if q == 19 else 200.0) * nodes * c["steps"]}
    if c["kind"] == "sweep":
        nodes = float(I.tube_sweep(c["tubes"])[0].sum())
        return {"bytes": 11 * 8.0 * nodes, "flops": 440.0 * nodes * c["steps"]}
    # forward, recompute and reverse (about three updates' work) of g
    return {"bytes": (5 + 4 + 1) * 8.0 * c["nx"], "flops": 3 * 300.0 * c["nx"] * c["steps"]}


# ----------------------------------------------------------------------------- 64-bit statement of the scheme
def _links(d2):
    if d2:
        c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
    else:
        c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
             (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
             (0, 1, -1), (0, -1, 1)]
        w = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    C = torch.tensor(c, dtype=torch.float64, device=DEV)
    return C, torch.tensor([w[sum(abs(v) for v in a)] for a in c], dtype=torch.float64, device=DEV)


class _Scheme:
    """States f, g of shape (Q, nodes); taus are numbers or per-node tensors."""

    def __init__(self, shape, bc, d2=False, collision="mrt", tau_f=0.9, tau_v=0.9, tau_e=0.9, tau_eps=0.9, tau_q=None,
                 eta=0.0, c7=0.0, sources=None):
        self.C, self.W = _links(d2)
        self.Q, self.d2, self.mrt, self.eta, self.c7 = len(self.W), d2, collision == "mrt", eta, c7
        self.tau = (tau_f, tau_v, tau_e, tau_eps, tau_q)
        nz, ny, nx = shape
        self.shape = shape

        def src(n, c, b):
            i = torch.arange(n, device=DEV) - c
            return i.clamp(0, n - 1) if b == ZG else i % n
        self.axis = [{k: src(n, k, b) for k in (-1, 0, 1)} for n, b in zip((nx, ny, nz), bc)]
        self.sources = sources
        if sources is None and nx * ny * nz < 3e7:
            self.sources = [((self.axis[2][int(c[2])][:, None, None] * ny + self.axis[1][int(c[1])][None, :, None]) * nx
                             + self.axis[0][int(c[0])][None, None, :]).reshape(-1) for c in self.C.tolist()]
        # rows of the moment matrix whose rates differ from tau_v, with their squared norms
        c2 = (self.C ** 2).sum(1)
        if d2:
            rows = [3 * c2 - 4, (9 * c2 * c2 - 21 * c2 + 8) / 2] + [(3 * c2 - 5) * self.C[:, i] for i in range(2)]
        else:
            rows = [19 * c2 - 30, (21 * c2 * c2 - 53 * c2 + 24) / 2] + [(5 * c2 - 9) * self.C[:, i] for i in range(3)]
        self.R = torch.stack(rows)
        self.R2 = (self.R ** 2).sum(1)

    def equilibria(self, N0, sigma, P, u):
        u2, cu = (u * u).sum(0), self.C @ u
        poly = 3 * cu + 4.5 * cu * cu - 1.5 * u2
        W = self.W[:, None]
        geq = W * (3 * P + sigma * poly)
        s = geq[1:].sum(0)
        return W * N0 * (1 + poly), torch.cat([(sigma - P - s)[None], geq[1:]])

    def recover(self, f, g):
        N0, T, M = f.sum(0), g.sum(0), self.C.T @ g
        u = 3 * M / (2 * T + torch.sqrt(4 * T * T - 3 * (M * M).sum(0)))
        sigma = 4 * T / (3 + (u * u).sum(0))
        return N0, sigma, sigma - T, u

    def init(self, e, ux, uy, uz, n):
        u = torch.stack([ux, uy, uz]).reshape(3, -1)
        g2 = 1 / (1 - (u * u).sum(0))
        e, n = e.reshape(-1), n.reshape(-1)
        return self.equilibria(n * torch.sqrt(g2), 4 / 3 * e * g2, e / 3, u)

    def pull(self, p):
        return torch.stack([p[a][self.sources[a]] for a in range(self.Q)])

    def step(self, f, g):
        f, g = self.pull(f), self.pull(g)
        N0, sigma, P, u = self.recover(f, g)
        feq, geq = self.equilibria(N0, sigma, P, u)
        tf, tv, te, tp, tq = self.tau
        if self.eta:
            ig = torch.sqrt(1 - (u * u).sum(0))
            n = N0 * ig
            T = P / n
            s = n * (4 - torch.log(n / (16 / math.pi ** 2 * T ** 3)))
            tg = 0.5 + self.eta * s * ig / (4 / 3 * P)
            te, tp, tq = (0.5 + a * (tg - 0.5) for a in (te, tp, tq if tq else 1.0))
            tf, tv = tf if tf and tf > 0 else tg, tg
        d = g - geq
        out = g - d / tv
        if self.mrt:
            tq = tv if tq is None else tq
            m = (self.R @ d) / self.R2[:, None]
            rates = [1 / te - 1 / tv, 1 / tp - 1 / tv] + [1 / tq - 1 / tv] * (len(self.R) - 2)
            for k, r in enumerate(rates):
                out = out - (r * m[k]) * self.R[k][:, None]
        if self.c7:
            out = out + self.correction(sigma, P, u, tv)
        return f - (f - feq) / tf, out

    def correction(self, sigma, P, u, tv):
        gam = 1 / torch.sqrt(1 - (u * u).sum(0))
        theta = 1 + 1 / (4 * gam * gam - 1)
        nz, ny, nx = self.shape

        def diff(v, a):
            v = v.reshape(ny, nx)
            return (0.5 * (v.index_select(1 - a, self.axis[a][-1]) - v.index_select(1 - a, self.axis[a][1]))).reshape(-1)

        def E(a):
            w = u[a]
            return 2 * (w * diff(sigma / 3 - P, a) - sigma / 3 * w * diff(gam, a) / gam - w * diff(sigma * w * w, a)) \
                + self.c7 * w * w * theta * diff(sigma * w, a)
        dq = 0.25 * (1 - 0.5 / tv) * (E(0) - E(1))
        return (self.C[:, 0] ** 2 - self.C[:, 1] ** 2)[:, None] * ((self.C ** 2).sum(1) == 1)[:, None] * dq

    def fields(self, f, g, shape):
        N0, _, P, u = self.recover(f, g)
        n = N0 * torch.sqrt(1 - (u * u).sum(0))
        if self.shape[:2] == (1, 1):   # a tube along x: nothing moves across it
            u = torch.stack([u[0], torch.zeros_like(u[0]), torch.zeros_like(u[0])])
        return {k: v.reshape(shape) for k, v in zip(FIELDS, (3 * P, P, u[0], u[1], u[2], n))}


def _exact_run(c, seed):
    shape = (c["nz"], c["ny"], c["nx"])
    tq = c["tau_q"] if c["tau_q"] > 0 else None
    s = _Scheme(shape, (c["bcx"], c["bcy"], c["bcz"]), c["lattice"] == "d2q9", c["collision"], c["tau_f"], c["tau_v"],
                c["tau_e"], c["tau_eps"], tq, c["eta"], {"": 0.0, "c7": 1.0, "c7_printed": 2.0}[c["correction"]])
    f, g = s.init(*_fields(c, seed))
    for _ in range(c["steps"]):
        f, g = s.step(f, g)
    out = s.fields(f, g, shape)
    if c["totals"]:
        out["totals"] = [float(f.sum()), float(g.sum())]
    if c["state"]:
        out["state"] = torch.cat([f, g]).reshape((2 * s.Q,) + shape)
    return out


def _exact_sweep(c, seed):
    lengths, taus, fields = _sweep_inputs(c, seed)
    lens = torch.from_numpy(lengths.astype(np.int64)).to(DEV)
    first = torch.repeat_interleave(torch.cumsum(lens, 0) - lens, lens)
    last = first + torch.repeat_interleave(lens, lens) - 1
    node = torch.arange(len(first), device=DEV)
    near = {k: torch.minimum(torch.maximum(node - k, first), last) for k in (-1, 0, 1)}
    tv, te, tp = torch.repeat_interleave(torch.from_numpy(taus).to(DEV), lens, dim=0).T
    s = _Scheme((1, 1, 1), (PER, PER, PER), False, "mrt", tv, tv, te, tp,
                sources=[near[int(a[0])] for a in _links(False)[0].tolist()])
    f, g = s.init(*fields)
    for _ in range(c["steps"]):
        f, g = s.step(f, g)
    return s.fields(f, g, (-1,))


def _exact_grad(c, seed):
    e, ux, uy, uz, n = _fields(c, seed)
    tgt = [t.reshape(-1) for t in _targets(c, seed)]
    taus = [torch.tensor(c[k], dtype=torch.float64, device=DEV, requires_grad=True) for k in ("tau_v", "tau_e", "tau_eps")]
    e0 = e.detach().requires_grad_(True)
    s = _Scheme((1, 1, c["nx"]), (ZG, PER, PER), False, c["collision"], c["tau_v"], *taus)
    f, g = s.init(e0, ux, uy, uz, n)
    f = f.detach()   # the misfit does not depend on f
    for _ in range(c["steps"]):
        g = s.step(f, g)[1]
    _, _, P, u = s.recover(f, g)
    loss = ((P - tgt[0]) ** 2).sum() + sum(((u[k] - tgt[1 + k]) ** 2).sum() for k in range(3))
    grads = torch.autograd.grad(loss, [*taus, e0], allow_unused=True)
    dtau = torch.stack([d if d is not None else torch.zeros((), dtype=torch.float64, device=DEV) for d in grads[:3]])
    loss = loss.detach()
    return {"loss": float(loss) if c["kind"] == "grad" else loss, "dtau": dtau, "de0": grads[3]}


def exact(case, seed):
    c = case
    if c["kind"] == "run":
        nodes = c["nx"] * c["ny"] * c["nz"]
        # the largest lattices take more time (and memory) than is worth it in plain torch
        return None if nodes > 3e7 or nodes * c["steps"] > 1e9 else _exact_run(c, seed)
    return _exact_sweep(c, seed) if c["kind"] == "sweep" else _exact_grad(c, seed)
