"""The work whose speed is measured, as a user's program asks for it.

Each case is one call sequence through the public Python binding
(paper_2608_26908_gb300.gpflbm.Sim), on inputs that are on the GPU already:

* ``steps``   -- load a state (phi, mu, f), advance it n time steps, read the
  whole state and the velocity back: the pass of a parameter scan, or of a run
  between two outputs;
* ``adjoint`` -- J and its gradients after a horizon of steps through the
  torch.autograd.Function: one iteration of an optimisation loop;
* ``totals``  -- the conservation totals and the derived fields (c, rho, u) of
  a loaded state: what a monitored run asks for between two batches of steps.

The named workloads, their sizes and their parameters are those of
paper_2608_26908_gb300/inputs.py; the inputs are grown states rather than the
workloads' first ones (a diffuse interface, a melt in motion, solute around
the solid), since a run spends nearly all of its steps on those.

``exact`` is the model restated in plain torch in 64 bits, for whole arrays.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2608_26908_gb300 import gpflbm, inputs

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"

# the objective of the differentiation workload (seed centre: the grid's)
W_FRAC, W_TIP, KAPPA = 1.0, 1.0, 2.0


def listed():
    return [
        # The single dendrite in FP64 on its own grid: a small problem run for
        # accuracy, thousands of steps, far too small to fill the chip.
        dict(name="dendrite2d-fp64", kind="steps", workload="dendrite2d", nx=128, ny=128, nz=1,
             precision="fp64", lattice=9, steps=100, solid=10.0, model="plain"),
        # The smallest call: one step of a small box between two reads, as an
        # interactive session or a coupled code does; latency is all of it.
        dict(name="dendrite2d-one-step", kind="steps", workload="dendrite2d", nx=70, ny=52, nz=1,
             precision="fp32", lattice=9, steps=1, solid=6.0, model="plain"),
        # The 2D eutectic workload at its own size.
        dict(name="eutectic2d", kind="steps", workload="eutectic2d", nx=1024, ny=512, nz=1,
             precision="fp32", lattice=9, steps=100, solid=64.0, model="plain"),
        # A grown dendrite on the paper's own odd-sized 2D domain.
        dict(name="dendrite2d-1001", kind="steps", workload="dendrite2d", nx=1001, ny=1001, nz=1,
             precision="fp32", lattice=9, steps=64, solid=150.0, model="plain"),
        # Directional growth with the shrinkage flow the paper switches on
        # (its 700-row domains; a width no tile divides).
        dict(name="eutectic2d-shrinkage", kind="steps", workload="eutectic2d", nx=500, ny=700, nz=1,
             precision="fp32", lattice=9, steps=50, solid=200.0, model="shrinkage"),
        # The 3D dendrite workload, populations in FP32 and in FP16.
        dict(name="dendrite3d", kind="steps", workload="dendrite3d", nx=256, ny=256, nz=256,
             precision="fp32", lattice=19, steps=20, solid=24.0, model="plain"),
        dict(name="dendrite3d-f16", kind="steps", workload="dendrite3d", nx=256, ny=256, nz=256,
             precision="fp32_f16", lattice=19, steps=20, solid=24.0, model="plain"),
        # The ternary eutectic workload at its own size, early in the run ...
        dict(name="eutectic3d", kind="steps", workload="eutectic3d", nx=256, ny=256, nz=512,
             precision="fp32", lattice=19, steps=10, solid=24.0, model="plain"),
        # ... and a smaller ragged box half filled with grains, late in one.
        dict(name="eutectic3d-grown", kind="steps", workload="eutectic3d", nx=150, ny=130, nz=171,
             precision="fp32", lattice=19, steps=20, solid=80.0, model="plain"),
        # The paper's own 3D lattice, crystal axes turned.
        dict(name="dendrite3d-q27-tilt", kind="steps", workload="dendrite3d", nx=120, ny=120, nz=120,
             precision="fp32", lattice=27, steps=20, solid=20.0, model="tilt"),
        # Backward: the differentiation workload's gradient.
        dict(name="adjoint2d", kind="adjoint", workload="adjoint2d", nx=512, ny=512, nz=1,
             precision="fp32", lattice=9, steps=200, ckpt=50, solid=40.0, model="plain"),
        # What a monitored run reads between two batches of steps.
        dict(name="eutectic3d-totals", kind="totals", workload="eutectic3d", nx=256, ny=256, nz=256,
             precision="fp32", lattice=19, steps=0, solid=60.0, model="plain"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["2d", "2d", "2d-fp64", "3d", "3d", "3d", "adjoint", "totals"])
    model = rng.choice(["plain", "plain", "plain", "shrinkage", "tilt", "ceqT"])
    if kind in ("2d", "2d-fp64"):
        fp64 = kind == "2d-fp64"
        nx, ny = _spread(rng, 48, 200 if fp64 else 1100), _spread(rng, 48, 200 if fp64 else 1100)
        name = rng.choice(["dendrite2d", "eutectic2d"])
        solid = _spread(rng, 6, max(7, 0.3 * min(nx, ny)))
        return dict(kind="steps", workload=name, nx=nx, ny=ny, nz=1, precision="fp64" if fp64 else "fp32",
                    lattice=9, steps=_spread(rng, 1, 100), solid=float(solid), model=model)
    if kind == "adjoint":
        nx, ny = _spread(rng, 64, 520), _spread(rng, 64, 520)
        steps = _spread(rng, 20, 120)
        return dict(kind="adjoint", workload="adjoint2d", nx=nx, ny=ny, nz=1,
                    precision=rng.choice(["fp32", "fp32", "fp32", "fp64"]) if nx * ny < 40000 else "fp32",
                    lattice=9, steps=steps, ckpt=_spread(rng, 5, steps), solid=float(_spread(rng, 8, 0.25 * min(nx, ny))),
                    model="plain")
    nx, ny, nz = (_spread(rng, 40, 256) for _ in range(3))
    name = rng.choice(["dendrite3d", "eutectic3d"])
    top = 0.3 * min(nx, ny, nz) if name == "dendrite3d" else 0.5 * nz
    solid = float(_spread(rng, 8, max(9, top)))
    if kind == "totals":
        return dict(kind="totals", workload=name, nx=nx, ny=ny, nz=nz,
                    precision=rng.choice(["fp32", "fp32", "fp32_f16"]), lattice=19, steps=0, solid=solid,
                    model="plain")
    lattice = rng.choice([19, 19, 19, 27])
    precision = rng.choice(["fp32", "fp32", "fp32_f16", "fp32_bf16"]) if lattice == 19 else "fp32"
    steps = max(1, min(20, int(4e7 / (nx * ny * nz))))
    return dict(kind="steps", workload=name, nx=nx, ny=ny, nz=nz, precision=precision, lattice=lattice,
                steps=_spread(rng, 1, steps), solid=solid, model=model)


# ---------------------------------------------------------------- inputs
def _scenario(case):
    sc = inputs.scenario(case["workload"], nx=case["nx"], ny=case["ny"], nz=case["nz"],
                         precision=case["precision"])
    sc["grid"]["nz"] = case["nz"]
    sc["grid"]["lattice"] = case["lattice"]
    p, NP = sc["params"], sc["n_phases"]
    if case["model"] == "shrinkage":
        p["eta_rho"] = [0.0] + [0.2] * (NP - 1) + [0.0] * (4 - NP)
    elif case["model"] == "tilt":
        for a in range(1, NP):
            p["tilt"][0][a] = p["tilt"][a][0] = 0.3
    elif case["model"] == "ceqT":
        for a in range(NP):
            p["dceq_dT"][a] = [0.1 * (a + 1), 0.05 * (a + 1)]
        p["G"], p["V"] = p["G"] or 1e-4, p["V"] or 1e-3
    return sc


def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if case["nz"] > 1 else (case["ny"], case["nx"])


def _modes(gen, shape, count=3):
    """A smooth random field of order one: a few long periodic waves."""
    out = torch.zeros(shape, dtype=torch.float64, device=DEVICE)
    r = torch.rand((count, len(shape) + 2), generator=gen, device=DEVICE, dtype=torch.float64).tolist()
    for row in r:
        arg = torch.zeros((1,) * len(shape), dtype=torch.float64, device=DEVICE)
        for a, n in enumerate(shape):
            x = torch.arange(n, dtype=torch.float64, device=DEVICE) * (2.0 * math.pi * (1 + int(3 * row[a])) / n)
            arg = arg + x.reshape([-1 if b == a else 1 for b in range(len(shape))])
        out += (0.5 + row[-2]) / count * torch.sin(arg + 2.0 * math.pi * row[-1])
    return out


def _blur(t, dims, passes):
    """Three-cell means along the grid axes, mirrored at the ends: turns sharp
    indicators into interfaces a few cells wide; ones and zeros stay exact."""
    for _ in range(passes):
        for d in dims:
            n = t.shape[d]
            lo = torch.cat([t.narrow(d, 0, 1), t.narrow(d, 0, n - 1)], d)
            hi = torch.cat([t.narrow(d, 1, n - 1), t.narrow(d, n - 1, 1)], d)
            t = (lo + t + hi) / 3.0
    return t


def _phases(case, sc, gen):
    shape, NP = _shape(case), sc["n_phases"]
    D = len(shape)
    eps = sc["params"]["eps"]
    ax = [torch.arange(n, dtype=torch.float64, device=DEVICE).reshape([-1 if b == a else 1 for b in range(D)])
          for a, n in enumerate(shape)]
    if sc["init"]["kind"] == "seed":
        jit = torch.rand(D, generator=gen, device=DEVICE, dtype=torch.float64).tolist()
        rel = [ax[a] + 0.5 - shape[a] / 2.0 - 3.0 * (jit[a] - 0.5) for a in range(D)]
        r2 = sum(v * v for v in rel)
        r4 = sum(v ** 4 for v in rel)
        # four (six) arms along the axes
        radius = case["solid"] * (1.0 + 0.15 * (4.0 * r4 / (r2 * r2 + 1e-9) - 3.0))
        half = math.pi ** 2 * eps / 8.0
        d = torch.clamp(torch.sqrt(r2) - radius, -half, half)
        s = 0.5 * (1.0 - torch.sin(4.0 * d / (math.pi * eps)))
        return torch.stack([1.0 - s, s])
    plane = shape[1:]
    if sc["init"]["kind"] == "lamellae":
        off = int(torch.randint(0, 32, (1,), generator=gen, device=DEVICE))
        which = 1 + ((torch.arange(shape[1], device=DEVICE) + off) // sc["init"]["width"]) % 2
    else:
        n = max(3, int(round(plane[0] * plane[1] / (math.pi * (sc["init"]["diameter"] / 2.0) ** 2))))
        at = torch.rand((3, n), generator=gen, device=DEVICE, dtype=torch.float64)
        owner = torch.full(plane, 1e30, dtype=torch.float64, device=DEVICE)
        which = torch.zeros(plane, dtype=torch.int64, device=DEVICE)
        for s0 in range(0, n, 64):
            dy = (ax[1][0] + 0.5)[None] - (at[0, s0:s0 + 64] * plane[0])[:, None, None]
            dx = (ax[2][0] + 0.5)[None] - (at[1, s0:s0 + 64] * plane[1])[:, None, None]
            dy, dx = dy.abs(), dx.abs()
            dy, dx = torch.minimum(dy, plane[0] - dy), torch.minimum(dx, plane[1] - dx)
            d2, k = (dy * dy + dx * dx).min(dim=0)
            ph = 1 + torch.clamp((at[2, s0:s0 + 64] * 3).to(torch.int64), max=2)
            which = torch.where(d2 < owner, ph[k], which)
            owner = torch.minimum(d2, owner)
    top = case["solid"] + 2.0 * _modes(gen, plane)
    solid = ax[0] + 0.5 < top
    phi = torch.stack([(solid & (which == a)) if a else ~solid for a in range(NP)]).to(torch.float64)
    return _blur(phi, range(1, D + 1), 2)


def _velocities(q):
    if q == 9:
        c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
        return c, w
    c = [(0, 0, 0)]
    for a in range(3):
        for s in (1, -1):
            c.append(tuple(s if b == a else 0 for b in range(3)))
    for a, b in ((0, 1), (0, 2), (1, 2)):
        for s, t in ((1, 1), (-1, -1), (1, -1), (-1, 1)):
            v = [0, 0, 0]
            v[a], v[b] = s, t
            c.append(tuple(v))
    if q == 19:
        return c, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    for v in ((1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)):
        c += [v, tuple(-x for x in v)]
    return c, [8 / 27] + [2 / 27] * 6 + [1 / 54] * 12 + [1 / 216] * 8


def _inputs(case, seed):
    """(phi, mu, f) of the exchange type on DEVICE, flat planes, from the seed."""
    sc = _scenario(case)
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed))
    shape, NP, NC = _shape(case), sc["n_phases"], sc["n_solutes"]
    D = len(shape)
    tdtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    phi = _phases(case, sc, gen)
    liquid = phi[0]
    # rejected solute along the solid, long waves in the melt, noise
    near = 4.0 * liquid * (1.0 - liquid)
    mu = torch.stack([0.02 * _modes(gen, shape) + 0.03 * near for _ in range(NC)])
    mu += 1e-3 * (2.0 * torch.rand(mu.shape, generator=gen, device=DEVICE, dtype=torch.float64) - 1.0)
    f = None
    if case["kind"] != "adjoint":
        c, w = _velocities(case["lattice"])
        u = [2e-3 * liquid * _modes(gen, shape) for _ in range(D)]
        drho = 1e-4 * _modes(gen, shape)
        uu = sum(v * v for v in u)
        f = torch.empty((len(c),) + shape, dtype=tdtype, device=DEVICE)
        for k in range(len(c)):
            cu = sum(c[k][a] * u[a] for a in range(D)) + torch.zeros_like(uu)
            f[k] = (w[k] * (1.0 + drho) * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)).to(tdtype)
        f = f.reshape(-1)
    return sc, phi.to(tdtype).reshape(-1), mu.to(tdtype).reshape(-1), f


def prepare(case, seed):
    sc, phi, mu, f = _inputs(case, seed)
    state = {"case": case, "phi": phi, "mu": mu, "f": f, "sim": gpflbm.Sim(sc)}
    if case["kind"] == "totals":
        state["sim"].set_state(phi, mu, f)
    elif case["kind"] == "adjoint":
        state["obj"] = dict(w_frac=W_FRAC, w_tip=W_TIP, kappa=KAPPA, x0=case["nx"] // 2, y0=case["ny"] // 2)
        p = sc["params"]
        state["leaves"] = [torch.tensor(v, dtype=torch.float64, requires_grad=True)
                           for v in (1.0 / p["tau_phi"], p["delta"][0][1], p["gbeta_c"][0])]
    return state


def run(state):
    case, sim = state["case"], state["sim"]
    if case["kind"] == "steps":
        sim.set_state(state["phi"], state["mu"], state["f"])
        sim.step(case["steps"])
        return sim.fields(("phi", "mu", "f", "u"), device=True)
    if case["kind"] == "adjoint":
        mu0 = state["mu"].detach().requires_grad_(True)
        J = gpflbm.GPFLBMFunction().apply(mu0, *state["leaves"], sim, state["phi"], state["obj"], case["steps"],
                                          case["ckpt"])
        grads = torch.autograd.grad(J, [mu0] + state["leaves"])
        return {"J": J.detach(), "mu0": grads[0], "mobility": grads[1], "delta": grads[2], "gbeta": grads[3]}
    mass, solute, solid, _ = sim.invariants()
    out = sim.fields(("c", "rho", "u"), device=True)
    out.update(mass=mass, solute=solute, solid=solid)
    return out


def work(case):
    """Bytes: every step reads and writes the stored state once (stored
    planes: one phase plane for two phases, all of them otherwise), the load
    and the read-back their planes.  Flops: the collision, the solute faces
    and the update of a melt cell, which no cell can do without; an adjoint
    step costs about two of them and the stored forward states are read back
    and rebuilt once."""
    sc = _scenario(case)
    cells = case["nx"] * case["ny"] * case["nz"]
    D, Q, NP, NC = (3 if case["nz"] > 1 else 2), case["lattice"], sc["n_phases"], sc["n_solutes"]
    real = 8 if case["precision"] == "fp64" else 4
    store = 2 if case["precision"] in ("fp32_f16", "fp32_bf16") else real
    state = Q * store + ((1 if NP == 2 else NP) + NC) * real
    flops = 12 * Q + 14 * D * (1 + NC)
    exchange = (NP + NC + Q) * real
    if case["kind"] == "steps":
        n = case["steps"]
        return {"bytes": cells * (2.0 * n * state + 2 * (exchange + state) + D * real), "flops": cells * float(n * flops)}
    if case["kind"] == "adjoint":
        n = case["steps"]
        # forward, rebuilt segments, and backward: the stored state and the
        # adjoint state read, the adjoint state written
        return {"bytes": cells * float(n) * (2 * state + 2 * state + 3 * state), "flops": cells * float(n) * 4 * flops}
    return {"bytes": cells * (2.0 * state + (NC + 1 + D) * real), "flops": cells * 4.0 * Q}


# ---------------------------------------------------------------- exact
class _Model:
    """The time step on whole arrays in 64 bits; axis a of the grid (0 = x) is
    dimension -1 - a of the arrays, one array per phase, solute, population."""

    def __init__(self, sc, shape, leaves=None):
        self.sc, self.p, self.shape, self.D = sc, sc["params"], shape, len(shape)
        self.NP, self.NC = sc["n_phases"], sc["n_solutes"]
        self.c, self.w = _velocities(sc["grid"]["lattice"])
        p = self.p
        self.mob = (leaves[0] if leaves else 1.0 / p["tau_phi"]) / p["eps"]
        self.delta = [row[:] for row in p["delta"]]
        if leaves:
            self.delta[0][1] = self.delta[1][0] = leaves[1]
        self.gb = list(p["gbeta_c"])
        if leaves:
            self.gb[0] = leaves[2]
        self.wall = [sc["grid"]["bc"][a] == inputs.WALL for a in range(self.D)]
        self.inv2A = [1.0 / (2.0 * a) for a in p["A"]]
        obs = torch.zeros(shape, dtype=torch.bool, device=DEVICE)
        for a in range(self.D):
            r, n = sc["grid"]["wall_rows"][a], shape[-1 - a]
            if r:
                obs.narrow(-1 - a, 0, r).fill_(True)
                obs.narrow(-1 - a, n - r, r).fill_(True)
        self.obs = obs if bool(obs.any()) else None
        n = shape[0]
        self.v = torch.arange(n, dtype=torch.float64, device=DEVICE).reshape([-1] + [1] * (self.D - 1))
        self.open = []
        for a in range(self.D):
            m = torch.ones(shape, dtype=torch.bool, device=DEVICE)
            if self.wall[a]:
                m.narrow(-1 - a, shape[-1 - a] - 1, 1).fill_(False)
            self.open.append(m)
        self.aniso = any(sc["params"]["delta"][a][b] != 0.0 or p["tilt"][a][b] != 0.0
                         for a in range(self.NP) for b in range(self.NP) if a != b)

    def nb(self, t, a, s):
        """The value of the neighbour at +s (1 or -1) along axis a."""
        d = t.dim() - 1 - a
        if not self.wall[a]:
            return torch.roll(t, -s, d)
        n = t.shape[d]
        if s > 0:
            return torch.cat([t.narrow(d, 1, n - 1), t.narrow(d, n - 1, 1)], d)
        return torch.cat([t.narrow(d, 0, 1), t.narrow(d, 0, n - 1)], d)

    def theta(self, t):
        p = self.p
        return -p["undercool"] + p["G"] * (self.v - p["v0"] - p["V"] * t)

    def ceq(self, a, i, th):
        k = self.p["dceq_dT"][a][i]
        return self.p["ceq"][a][i] + (k * th if k else 0.0)

    def h(self, ph, a):
        s = 0.0
        for b in range(self.NP):
            for g in range(b + 1, self.NP):
                if b != a and g != a:
                    s = s + ph[b] * ph[g]
        return ph[a] * ph[a] * (3.0 - 2.0 * ph[a]) + 2.0 * ph[a] * s

    def dh(self, ph, b, a):
        if a == b:
            s = 0.0
            for g in range(self.NP):
                for d in range(g + 1, self.NP):
                    if g != b and d != b:
                        s = s + ph[g] * ph[d]
            return 6.0 * ph[b] * (1.0 - ph[b]) + 2.0 * s
        s = 0.0
        for d in range(self.NP):
            if d != a and d != b:
                s = s + ph[d]
        return 2.0 * ph[b] * s

    def dA(self, a, b, q, want):
        """Components `want` of dA/dq of the pair (a, b)."""
        delta, floor = self.delta[a][b], self.p["q_floor"]
        if isinstance(delta, float) and delta == 0.0:
            return [2.0 * q[j] for j in want]
        th = self.p["tilt"][a][b]
        cs, sn = math.cos(th), math.sin(th)
        r = q if th == 0.0 else [cs * q[0] + sn * q[1], cs * q[1] - sn * q[0]] + q[2:]
        s2 = sum(v * v for v in r)
        s4 = sum(v ** 4 for v in r)
        small = s2 <= floor
        inv2 = 1.0 / torch.where(small, torch.ones_like(s2), s2)
        ac = 1.0 - delta * (3.0 - 4.0 * s4 * inv2 * inv2)

        def comp(j):
            dac = 16.0 * delta * (r[j] ** 3 - r[j] * s4 * inv2) * inv2 * inv2
            return torch.where(small, 2.0 * r[j], 2.0 * ac * (ac * r[j] + s2 * dac))

        if th == 0.0:
            return [comp(j) for j in want]
        d = {j: comp(j) for j in set(want) | {0, 1}}
        turn = {0: lambda: cs * d[0] - sn * d[1], 1: lambda: sn * d[0] + cs * d[1], 2: lambda: d[2]}
        return [turn[j]() for j in want]

    def phase_field(self, ph, mu, th):
        NP, D, p = self.NP, self.D, self.p
        zero = torch.zeros(self.shape, dtype=torch.float64, device=DEVICE)
        div = [zero] * NP
        for d in range(D):
            up = [self.nb(v, d, 1) for v in ph]
            pf = [0.5 * (a + b) for a, b in zip(ph, up)]
            g = []
            for a in range(NP):
                row = [None] * D
                row[d] = up[a] - ph[a]
                for t in range(D):
                    if t != d and self.aniso:
                        s = ph[a] + up[a]
                        row[t] = 0.25 * (self.nb(s, t, 1) - self.nb(s, t, -1))
                g.append(row)
            fl = [zero] * NP
            for a in range(NP):
                for b in range(a + 1, NP):
                    gab = p["gamma"][a][b]
                    q = [pf[a] * g[b][t] - pf[b] * g[a][t] if g[a][t] is not None else zero for t in range(D)]
                    v = self.dA(a, b, q, [d])[0]
                    fl[a] = fl[a] - gab * pf[b] * v
                    fl[b] = fl[b] + gab * pf[a] * v
            for a in range(NP):
                x = torch.where(self.open[d], fl[a], zero)
                div[a] = div[a] + x - torch.roll(x, 1, -1 - d)
        gc = [[0.5 * (self.nb(v, t, 1) - self.nb(v, t, -1)) for t in range(D)] for v in ph]
        dad = [zero] * NP
        for a in range(NP):
            for b in range(a + 1, NP):
                gab = p["gamma"][a][b]
                q = [ph[a] * gc[b][t] - ph[b] * gc[a][t] for t in range(D)]
                v = self.dA(a, b, q, range(D))
                dad[a] = dad[a] + gab * sum(v[t] * gc[b][t] for t in range(D))
                dad[b] = dad[b] - gab * sum(v[t] * gc[a][t] for t in range(D))
        psi = []
        for b in range(NP):
            s = p["S"][b] * th
            for i in range(self.NC):
                s = s - (mu[i] * mu[i] / (4.0 * p["A"][b]) + mu[i] * self.ceq(b, i, th))
            psi.append(s)
        rate = []
        for a in range(NP):
            obst = sum(p["gamma"][a][b] * ph[b] for b in range(NP) if b != a)
            drv = sum(psi[b] * self.dh(ph, b, a) for b in range(NP))
            rate.append(p["eps"] * (div[a] - dad[a]) - 16.0 / (math.pi ** 2 * p["eps"]) * obst - drv)
        act = []
        for a in range(NP):
            m = (ph[a] > 0.0).to(torch.uint8)
            for x in range(D):
                m = torch.maximum(m, torch.maximum(self.nb(m, x, 1), self.nb(m, x, -1)))
            act.append(m > 0)
        na = sum(m.to(torch.float64) for m in act)
        multi = na >= 2.0
        if self.obs is not None:
            multi = multi & ~self.obs
        lam = sum(torch.where(m, r, zero) for m, r in zip(act, rate)) / na
        u = [ph[a] + self.mob * (rate[a] - lam) for a in range(NP)]
        if NP == 2:
            s = torch.where(multi, torch.clamp(u[1], 0.0, 1.0), ph[1])
            return [1.0 - s, s]
        low = torch.full(self.shape, -1e30, dtype=torch.float64, device=DEVICE)
        srt = torch.sort(torch.stack([torch.where(m, x, low) for m, x in zip(act, u)]), dim=0, descending=True)[0]
        run_, tau = zero, zero
        for j in range(NP):
            run_ = run_ + srt[j]
            t = (run_ - 1.0) / (j + 1)
            tau = torch.where((j < na) & (srt[j] - t > 0.0), t, tau)
        return [torch.where(multi, torch.where(m, torch.clamp(x - tau, min=0.0), zero), v)
                for m, x, v in zip(act, u, ph)]

    def macro(self, ph, mu, d, th, fs=None):
        """rho - 1, U, F of every cell (fs: the shrinkage force)."""
        p = self.p
        drho = sum(d)
        m = [sum(self.c[k][a] * d[k] for k in range(len(d)) if self.c[k][a]) for a in range(self.D)]
        phl = ph[0] if self.obs is None else torch.where(self.obs, torch.zeros_like(ph[0]), ph[0])
        kappa = 2.0 * (p["tau_f"] - 0.5) / 3.0 * p["h_drag"] / p["W0"] ** 2 * (1.0 - phl) ** 2
        drive = p["gbeta_T"] * (th + p["T_E"] - p["T_ref"])
        for i in range(self.NC):
            drive = drive + self.gb[i] * (self.ceq(0, i, th) - p["c_ref"][i] + mu[i] * self.inv2A[0])
        rho = 1.0 + drho
        force = [fs[a] if fs else 0.0 for a in range(self.D)]
        force[-1] = force[-1] + rho * phl * drive
        u = [(m[a] + 0.5 * force[a]) / (rho * (1.0 + 0.5 * kappa)) for a in range(self.D)]
        F = [force[a] - rho * kappa * u[a] for a in range(self.D)]
        return drho, u, F

    def collide(self, d, drho, u, F):
        it = 1.0 / self.p["tau_f"]
        pre = 1.0 - 0.5 * it
        rho = 1.0 + drho
        uu = sum(v * v for v in u)
        uF = sum(a * b for a, b in zip(u, F))
        post = []
        for k, c in enumerate(self.c):
            cu = sum(c[a] * u[a] for a in range(self.D) if c[a]) if any(c) else 0.0 * uu
            cF = sum(c[a] * F[a] for a in range(self.D) if c[a]) if any(c) else 0.0 * uu
            feq = drho + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
            g = 3.0 * (cF - uF) + 9.0 * cu * cF
            post.append((1.0 - it) * d[k] + self.w[k] * (it * feq + pre * g))
        return post

    def stream(self, post):
        opp = {c: k for k, c in enumerate(self.c)}
        out = []
        for k, c in enumerate(self.c):
            t = post[k]
            hit = torch.zeros((1,) * self.D, dtype=torch.bool, device=DEVICE)
            for a in range(self.D):
                if c[a]:
                    t = torch.roll(t, c[a], -1 - a)
                    if self.wall[a]:
                        n = self.shape[-1 - a]
                        row = torch.zeros(n, dtype=torch.bool, device=DEVICE)
                        row[0 if c[a] > 0 else n - 1] = True
                        hit = hit | row.reshape([-1 if x == self.D - 1 - a else 1 for x in range(self.D)])
            if any(c[a] and self.wall[a] for a in range(self.D)):
                t = torch.where(hit, post[opp[tuple(-x for x in c)]], t)
            out.append(t)
        return out

    def step(self, ph, mu, d, t):
        p, D, NP, NC = self.p, self.D, self.NP, self.NC
        zero = torch.zeros(self.shape, dtype=torch.float64, device=DEVICE)
        th = self.theta(t)
        pn = self.phase_field(ph, mu, th)
        fs = None
        if any(p["eta_rho"]):
            fs = [zero] * D
            for a in range(NP):
                if p["eta_rho"][a] == 0.0:
                    continue
                g = [0.5 * (self.nb(ph[a], x, 1) - self.nb(ph[a], x, -1)) for x in range(D)]
                g2 = sum(v * v for v in g)
                flat = g2 <= 1e-12
                s = torch.where(flat, zero, (pn[a] - ph[a]) / torch.sqrt(torch.where(flat, torch.ones_like(g2), g2)))
                fs = [fs[x] + p["eta_rho"][a] * s * g[x] for x in range(D)]
        drho, u, F = self.macro(ph, mu, d, th, fs)
        hl = self.h(pn, 0)
        M0 = p["D_liq"] * self.inv2A[0]
        div = [zero] * NC
        c0 = [self.ceq(0, i, th) + mu[i] * self.inv2A[0] for i in range(NC)]
        for x in range(D):
            nb = lambda v: self.nb(v, x, 1)  # noqa: E731
            up = [nb(v) for v in ph]
            Mf = 0.5 * M0 * (pn[0] + nb(pn[0]))
            ua = u[x] * hl
            J = [-Mf * (nb(mu[i]) - mu[i]) + 0.5 * (ua * c0[i] + nb(ua * c0[i])) for i in range(NC)]
            liq = 0.5 * (ph[0] + up[0])
            for a in range(1, NP):
                gn = up[a] - ph[a]
                s = ph[a] + up[a]
                g2 = gn * gn
                for y in range(D):
                    if y != x:
                        gt = 0.25 * (self.nb(s, y, 1) - self.nb(s, y, -1))
                        g2 = g2 + gt * gt
                flat = g2 <= 1e-12
                nd = torch.where(flat, zero, liq * gn / torch.sqrt(torch.where(flat, torch.ones_like(g2), g2)))
                rise = pn[a] - ph[a]
                dphi = 0.5 * (rise + nb(rise))
                for i in range(NC):
                    dc = p["ceq"][0][i] - p["ceq"][a][i]
                    k = p["dceq_dT"][0][i] - p["dceq_dT"][a][i]
                    if k:
                        tf = th + torch.zeros(self.shape, dtype=torch.float64, device=DEVICE)
                        dc = dc + k * 0.5 * (tf + nb(tf))
                    dc = dc + 0.5 * (mu[i] + nb(mu[i])) * (self.inv2A[0] - self.inv2A[a])
                    J[i] = J[i] - p["a_at"] * p["eps"] * dc * dphi * nd
            shut = ~self.open[x]
            if self.obs is not None:
                shut = shut | self.obs | nb(self.obs.to(torch.uint8)).to(torch.bool)
            for i in range(NC):
                f = torch.where(shut, zero, J[i])
                div[i] = div[i] + f - torch.roll(f, 1, -1 - x)
        hn = [self.h(pn, a) for a in range(NP)]
        ho = [self.h(ph, a) for a in range(NP)]
        chi = sum(hn[a] * self.inv2A[a] for a in range(NP))
        new = []
        for i in range(NC):
            src = zero
            for a in range(NP):
                src = src + (self.ceq(a, i, th) + mu[i] * self.inv2A[a]) * (hn[a] - ho[a])
                src = src - p["G"] * p["V"] * p["dceq_dT"][a][i] * hn[a]
            m = mu[i] + (-div[i] - src) / chi
            new.append(m if self.obs is None else torch.where(self.obs, mu[i], m))
        return pn, new, self.stream(self.collide(d, drho, u, F))


def _reference_state(case, sc, phi, mu, f):
    shape = _shape(case)
    ph = list(phi.double().reshape((sc["n_phases"],) + shape))
    m = list(mu.double().reshape((sc["n_solutes"],) + shape))
    _, w = _velocities(case["lattice"])
    if f is None:
        d = [torch.zeros(shape, dtype=torch.float64, device=DEVICE) for _ in w]
    else:
        d = [x.double() - w[k] for k, x in enumerate(f.reshape((len(w),) + shape))]
    return ph, m, d


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    sc, phi, mu, f = _inputs(case, seed)
    M = _Model(sc, _shape(case))
    with torch.no_grad():
        ph, m, d = _reference_state(case, sc, phi, mu, f)
        if sc["n_phases"] == 2:
            ph[0] = 1.0 - ph[1]  # the library keeps phi_1
        for t in range(case["steps"]):
            ph, m, d = M.step(ph, m, d, t)
        th = M.theta(case["steps"])
        drho, u, _ = M.macro(ph, m, d, th)
        u = torch.stack(u).reshape(M.D, -1)
        if case["kind"] == "steps":
            full = torch.stack([x + M.w[k] for k, x in enumerate(d)]).reshape(len(d), -1)
            return {"phi": torch.stack(ph).reshape(M.NP, -1), "mu": torch.stack(m).reshape(M.NC, -1), "f": full, "u": u}
        h = [M.h(ph, a) for a in range(M.NP)]
        c = [sum(h[a] * (M.ceq(a, i, th) + m[i] * M.inv2A[a]) for a in range(M.NP)) for i in range(M.NC)]
        cells = drho.numel()
        return {"c": torch.stack(c).reshape(M.NC, -1), "rho": (1.0 + drho).reshape(1, -1), "u": u,
                "mass": float(drho.sum()) + cells, "solute": np.array([float(v.sum()) for v in c]),
                "solid": float(sum(h[1:]).sum()) / cells}


def _exact_adjoint(case, seed):
    sc, phi, mu, _ = _inputs(case, seed)
    p = sc["params"]
    leaves = [torch.tensor(v, dtype=torch.float64, device=DEVICE, requires_grad=True)
              for v in (1.0 / p["tau_phi"], p["delta"][0][1], p["gbeta_c"][0])]
    ph, m, d = _reference_state(case, sc, phi, mu, None)
    s = ph[1]
    mu0 = m[0].clone().requires_grad_(True)

    def advance(t, mob, delta, gb, s, mu, *d):
        M = _Model(sc, _shape(case), [mob, delta, gb])
        a, b, c = M.step([1.0 - s, s], [mu], list(d), t)
        return (a[1], b[0]) + tuple(c)

    state = (s, mu0) + tuple(d)
    for t in range(case["steps"]):
        state = checkpoint(advance, t, *leaves, *state, use_reentrant=False)
    s = state[0]
    frac = (s * s * (3.0 - 2.0 * s)).mean()
    x0, y0, nx = case["nx"] // 2, case["ny"] // 2, case["nx"]
    r = torch.arange(nx - x0, dtype=torch.float64, device=DEVICE)
    tip = (r * torch.softmax(KAPPA * r * s[y0, x0:], 0)).sum()
    J = W_FRAC * frac + W_TIP * tip / nx
    g = torch.autograd.grad(J, [mu0] + leaves)
    return {"J": J.detach(), "mu0": g[0].reshape(-1), "mobility": g[1].cpu(), "delta": g[2].cpu(), "gbeta": g[3].cpu()}
