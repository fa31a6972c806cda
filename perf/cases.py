"""The timed cases of the sparse-lattice LBGK solver.

Each case is work that a program built on this package has it do, through its
public entry points (``hemegb.Solver``, ``validation.iolet_series``,
``adjoint.flow_objective``):

* ``flow``     a flow simulation's inner loop: advance some time steps, then read density,
               velocity and wall shear stress into device tensors (and, with ``check``, the
               FP64 mass and iolet fluxes that tell a diverging run);
* ``monitor``  the pulsatile pipe check: a tabulated heart beat drives the inlet, the iolet
               monitor is sampled every few steps;
* ``adjoint``  one gradient of a flow objective with respect to the relaxation time and the
               inlet amplitudes, as an optimiser's iteration takes it.

Lattices are the straight pipe and the seeded bifurcating vessel trees of this repository's
tests and benchmark, from the 12,352-site pipe to the 20M-site tree, in every storage
precision (FP32 by default; BF16 and FP16 for the large runs; FP64 for reference runs).  The
seed sets the initial velocity field, the phase of the inlet wave, the relaxation time and,
for the adjoint, the amplitudes and the targets; a vessel's geometry is a file on a user's
disk and does not depend on it.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2202_11770_gb300 import adjoint, geometry, hemegb, validation, workloads

ELEM = {"fp32": 4, "bf16": 2, "fp16": 2, "fp64": 8}


def _pipe(radius, length):
    return {"shape": "pipe", "radius": float(radius), "length": int(length)}


def _tree(sites, depth, shape_seed=2202):
    return {"shape": "tree", "sites": int(sites), "depth": int(depth), "shape_seed": int(shape_seed)}


def _flow(geom, steps, precision="fp32", scheme="auto", check=False, windkessel=False):
    return {"kind": "flow", **geom, "steps": int(steps), "precision": precision, "scheme": scheme, "check": bool(check),
            "windkessel": bool(windkessel)}


def listed():
    cases = {
        # the pipe of the paper's CPU/GPU comparison: the smallest lattice in use, launches count
        "pipe_12k_fp32": _flow(_pipe(8, 64), 200),
        # the same comparison's time series (flow, maximum velocity, pressure at the iolets) on a finer pipe
        "pipe_45k_monitor_fp32": {"kind": "monitor", **_pipe(12, 100), "steps": 200, "every": 20, "precision": "fp32",
                                  "scheme": "auto"},
        # a small vessel with downstream resistance models at its outlets
        "tree_50k_windkessel_fp32": _flow(_tree(50_000, 2), 100, windkessel=True),
        # a reference run in FP64, against which the other precisions are judged
        "tree_200k_fp64": _flow(_tree(200_000, 2, 11770), 40, "fp64"),
        # a vessel whose state fits the L2 cache, 16-bit storage
        "tree_500k_bf16": _flow(_tree(500_000, 6), 50, "bf16"),
        # a vessel past the L2 cache, an odd number of sites, an odd number of steps between read-outs
        "tree_1m_fp32": _flow(_tree(1_000_000, 4, 11770), 25),
        # the pull scheme by name (as partitioned runs use it), FP16, an odd number of sites
        "tree_2m_fp16_ab": _flow(_tree(2_000_000, 4, 11770), 20, "fp16", "ab"),
        # frequent snapshots with a divergence check: the read-out weighs as much as the steps
        "tree_8m_fp32_snapshot": _flow(_tree(8_000_000, 6), 2, check=True),
        # the benchmark's lattice, in its default form and in 16-bit storage
        "tree_20m_fp32": _flow(_tree(20_000_000, 6), 20),
        "tree_20m_bf16": _flow(_tree(20_000_000, 6), 20, "bf16"),
        # gradients on the small and on the benchmark's adjoint lattice, over long enough a run that the inlet's
        # pressure wave has passed the probe plane (the middle of the root vessel)
        "adjoint_50k_fp32": {"kind": "adjoint", **_tree(50_000, 2), "steps": 100, "precision": "fp32", "scheme": "auto"},
        "adjoint_2m_fp32": {"kind": "adjoint", **_tree(2_000_000, 4, 11770), "steps": 220, "precision": "fp32",
                            "scheme": "auto"},
    }
    return [{"name": k, **c} for k, c in cases.items()]


def _log_between(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(["flow", "monitor", "adjoint"], [14, 2, 4])[0]
    if kind == "monitor":
        every = rng.randint(5, 50)
        return {"kind": "monitor", **_pipe(rng.uniform(8.0, 24.0), rng.randint(50, 200)), "steps": every * rng.randint(4, 12),
                "every": every, "precision": rng.choice(["fp32", "fp32", "fp64"]), "scheme": rng.choice(["auto", "ab", "aa"])}
    if kind == "adjoint":
        sites = _log_between(rng, 30e3, 2e6)
        depth = 2 if sites < 300e3 else 4
        wave = (1.24 if depth == 2 else 1.05) * sites ** (1 / 3)   # steps from the inlet to the probe plane
        return {"kind": "adjoint", **_tree(sites, depth, rng.choice([2202, 11770])),
                "steps": int(wave * rng.uniform(1.3, 1.6)), "precision": "fp32", "scheme": "auto"}
    precision = rng.choices(["fp32", "bf16", "fp16", "fp64"], [10, 5, 3, 2])[0]
    scheme = rng.choices(["auto", "ab", "aa"], [6, 2, 2])[0]
    sites = _log_between(rng, 12e3, 2e6 if precision == "fp64" else 20e6)
    if sites < 1e6 and rng.random() < 0.3:
        radius = rng.uniform(6.0, min(60.0, (sites / 16.0 / math.pi) ** 0.5))
        geom = _pipe(radius, max(16, round(sites / (math.pi * radius * radius))))
        tree = False
    else:
        geom = _tree(sites, 2 if sites < 200e3 else 4 if sites < 4e6 else 6, rng.choice([2202, 11770]))
        tree = True
    steps = int(min(200, max(2, _log_between(rng, 10e6, 200e6) / sites)))
    return _flow(geom, steps, precision, scheme, rng.random() < 0.25, tree and sites < 1e6 and rng.random() < 0.15)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=3)
def _made(shape, *size):
    if shape == "pipe":
        return geometry.pipe(*size)
    sites, depth, shape_seed, sectors = size
    return workloads.tree_lattice(sites, depth=depth, seed=shape_seed, n_sectors=sectors, n_rings=sectors)


def _lattice(case):
    if case["shape"] == "pipe":
        return _made("pipe", case["radius"], case["length"])
    return _made("tree", case["sites"], case["depth"], case["shape_seed"], 8 if case["kind"] == "adjoint" else 1)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _inputs(case, seed, lattice):
    """What the seed decides, as plain values and (u0) a device tensor."""
    rng = np.random.default_rng(seed)
    pipe = case["shape"] == "pipe"
    tau = (0.8 if pipe else 0.55) + 0.02 * rng.uniform()
    if case["kind"] == "monitor":
        wave = validation.cardiac_waveform(period=400.0, peak=0.02 * (1.0 + 0.1 * rng.uniform(-1, 1)))
    else:
        wave = {"kind": "cosine", "mean": 0.01 if pipe else 0.02, "rel": 0.5, "period": 2000.0,
                "phase": float(rng.uniform(0, 2 * np.pi))}
    q = {"tau": float(tau), "wave": wave, "amps": np.ones(int(lattice.iolets[0].n_groups))}
    if case["kind"] == "adjoint":
        q["amps"] = (1.0 + 0.05 * rng.uniform(-1, 1, q["amps"].size)).astype(np.float32).astype(np.float64)
        q["tau"] = float(np.float32(q["tau"]))
        q["objective"] = workloads.root_midplane_objective(lattice, seed=seed)
        return q
    # a smooth velocity field of a few per mille of the speed of sound: eight waves along each axis
    dev = _device()
    x = torch.as_tensor(lattice.xyz, device=dev).T.to(torch.float32)
    u0 = torch.zeros((3, lattice.n), dtype=torch.float32, device=dev)
    for axis in range(3):
        k, phase, amp = rng.uniform(0.02, 0.2, 3), rng.uniform(0, 2 * np.pi, 3), 2e-3 * rng.normal(size=3)
        for a in range(3):
            u0[axis] += float(amp[a]) * torch.sin(float(k[a]) * x[a] + float(phase[a]))
    q["u0"] = u0
    if case.get("windkessel"):
        # resistances and compliances of the scale of the outlets' flow; every third outlet is a pure resistance
        q["wk"] = [(1e-4 * (1 + rng.uniform()), 0.0 if k % 3 == 2 else 2e4, 2e-4 * (1 + rng.uniform()), 1.0)
                   for k in range(len(lattice.iolets) - 1)]
    return q


def prepare(case, seed):
    lattice = _lattice(case)
    q = _inputs(case, seed, lattice)
    solver = hemegb.Solver(lattice, tau=q["tau"], precision=case["precision"], scheme=case["scheme"])
    for k in range(1, len(lattice.iolets)):
        solver.set_pressure(k, 1.0)
        if "wk" in q:
            solver.set_windkessel(k, *q["wk"][k - 1])
    state = {"case": case, "solver": solver}
    if case["kind"] == "adjoint":
        obj = q["objective"]
        state["objective"] = obj
        state["tau"] = torch.tensor(q["tau"], dtype=torch.float32, requires_grad=True)
        state["amps"] = torch.tensor(q["amps"], dtype=torch.float32, requires_grad=True)
        state["waves"] = {0: q["wave"]}
        state["workspace"] = solver.adjoint_workspace(case["steps"], obj.sites.size)
    else:
        solver.set_velocity(0, q["amps"], q["wave"])
        solver.init_equilibrium(1.0, q["u0"])
    return state


def run(state):
    case, solver = state["case"], state["solver"]
    if case["kind"] == "adjoint":
        obj, tau, amps = state["objective"], state["tau"], state["amps"]
        tau.grad = amps.grad = None
        loss = adjoint.flow_objective(tau, amps, solver, case["steps"], obj.sites, obj.target, obj.axis, state["waves"],
                                      workspace=state["workspace"])
        loss.backward()
        rho, u, _ = solver.macros_device(wss=False)
        return {"J": loss.detach(), "dtau": tau.grad, "damps": amps.grad, "rho": rho, "u": u}
    if case["kind"] == "monitor":
        series = validation.iolet_series(solver, case["steps"], case["every"])
        rho, u, _ = solver.macros_device(wss=False)
        return {"flux": series["flux"], "u_max": series["u_max"], "pressure": series["pressure"], "rho": rho, "u": u}
    solver.step(case["steps"])
    rho, u, wss = solver.macros_device()
    out = {"rho": rho, "u": u, "wss": wss}
    if case["check"]:
        out["mass"], out["flux"] = solver.reduce()
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """The populations are read once and written once a time step (19 values a site each way), and
    the read-out writes its fields; the streaming index is the solver's own table, so the least it
    could take is not counted.  A reverse step reads the state and the adjoint and writes the
    adjoint.  About 200 operations a site and step (400 for a reverse step)."""
    n, steps = _lattice(case).n, case["steps"]
    pop = 19 * ELEM[case["precision"]]
    if case["kind"] == "adjoint":
        return {"bytes": n * steps * (2 * pop + 3 * pop) + 16 * n, "flops": 600.0 * n * steps}
    if case["kind"] == "monitor":
        return {"bytes": n * steps * 2 * pop + 16 * n, "flops": 200.0 * n * steps}
    return {"bytes": n * steps * 2 * pop + 20 * n, "flops": 200.0 * n * steps}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
_C = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0], [-1, -1, 0],
               [1, -1, 0], [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1], [-1, 0, 1], [0, 1, 1], [0, -1, -1], [0, 1, -1],
               [0, -1, 1]])
_W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
_OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]


def _wave_at(w, t):
    if w["kind"] == "cosine":
        return w["mean"] * (1.0 + w["rel"] * math.cos(2.0 * math.pi * t / w["period"] + w["phase"]))
    s = w["samples"]
    pos = (t % w["period"]) / w["period"] * len(s)
    j = int(pos)
    return w["mean"] * ((1.0 - (pos - j)) * s[j % len(s)] + (pos - j) * s[(j + 1) % len(s)])


class _Plain:
    """The LBGK step on shifted populations h = f - w, [19, n] in FP64."""

    def __init__(self, lattice, tau, dev):
        self.lat, self.tau, self.dev, self.n = lattice, tau, dev, lattice.n
        n = self.n
        self.gather = []       # per direction: flat [19 n] source (fluid: row i at s; else row opp(i) at x)
        own = torch.arange(n, device=dev)
        links = {}
        for i in range(1, 19):
            s = torch.as_tensor(lattice.src[i - 1], device=dev).long()
            self.gather.append(torch.where(s >= 0, s + i * n, own + _OPP[i] * n))
            for x in torch.nonzero(s <= -2).ravel().cpu().numpy():
                links.setdefault(-int(lattice.src[i - 1, x]) - 2, []).append((i, int(x)))
        self.iolet = []        # (iolet, directions, sites, Ladd coefficient, group) of each iolet's links
        for k, pairs in sorted(links.items()):
            i, x = np.array(pairs).T
            io = lattice.iolets[k]
            c = _C[i].astype(np.float64)
            v = lattice.xyz[x] - 0.5 * c - io.centre
            r2 = ((v - (v @ io.normal)[:, None] * io.normal) ** 2).sum(1)
            coef = 6.0 * _W[i] * np.maximum(0.0, 1.0 - r2 / io.radius ** 2) * (c @ io.normal)
            t = lambda a, d: torch.as_tensor(a, dtype=d, device=dev)  # noqa: E731
            self.iolet.append({"k": k, "io": io, "i": t(i, torch.long), "x": t(x, torch.long), "c": t(c, torch.float64),
                               "w": t(_W[i], torch.float64), "coef": t(coef, torch.float64),
                               "group": t(lattice.amp_group[x], torch.long), "normal": t(io.normal, torch.float64)})

    @staticmethod
    def moments(h):
        drho = h.sum(0)
        rho = 1.0 + drho
        u = []
        for a in range(3):
            j = torch.zeros_like(drho)
            for i in range(1, 19):
                if _C[i, a]:
                    j = j + h[i] if _C[i, a] > 0 else j - h[i]
            u.append(j / rho)
        return drho, rho, u

    @staticmethod
    def heq(i, drho, rho, u, usq):
        cu = 0.0
        for a in range(3):
            if _C[i, a]:
                cu = cu + u[a] if _C[i, a] > 0 else cu - u[a]
        return _W[i] * (drho + rho * (3.0 * cu + 4.5 * cu * cu - usq))

    def equilibrium(self, u0):
        u = [u0[a].double() for a in range(3)]
        usq = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        zero, one = torch.zeros_like(usq), torch.ones_like(usq)
        return torch.stack([self.heq(i, zero, one, u, usq) for i in range(19)])

    def collide(self, h, tau):
        drho, rho, u = self.moments(h)
        usq = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        return torch.stack([h[i] + (self.heq(i, drho, rho, u, usq) - h[i]) / tau for i in range(19)])

    def stream(self, post, amps, val):
        """f(t+1) and each iolet's inflow, from s'(t); val[k]: w(t) or the ghost density."""
        flat = post.reshape(-1)
        h = torch.stack([post[0]] + [flat[g] for g in self.gather])
        flux = {}
        for L in self.iolet:
            i, x = L["i"], L["x"]
            out = h[i, x]                                  # s'_opp(i)(x)
            _, rho, u = self.moments(post[:, x])
            if L["io"].kind == geometry.VELOCITY:
                new = out + L["coef"] * rho * amps[L["group"]] * val[L["k"]]
            else:
                un = sum(u[a] * L["normal"][a] for a in range(3))
                g = [un * L["normal"][a] for a in range(3)]
                cu = sum(L["c"][:, a] * g[a] for a in range(3))
                usq = 1.5 * (g[0] ** 2 + g[1] ** 2 + g[2] ** 2)
                d = val[L["k"]] - 1.0
                new = L["w"] * (d + (1.0 + d) * (3.0 * cu + 4.5 * cu * cu - usq))
            h = h.index_put((i, x), new)
            flux[L["k"]] = float((new - out).sum().detach())
        return h, flux

    def wss(self, h):
        drho, rho, u = self.moments(h)
        usq = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        nrm = torch.as_tensor(self.lat.wall_normal, device=self.dev).double()
        tr = [torch.zeros_like(rho) for _ in range(3)]     # sum_i (f_i - feq_i) c_i (c_i . n)
        for i in range(1, 19):
            d = h[i] - self.heq(i, drho, rho, u, usq)
            cn = sum(float(_C[i, a]) * nrm[a] for a in range(3))
            for a in range(3):
                if _C[i, a]:
                    tr[a] = tr[a] + float(_C[i, a]) * cn * d
        k = -(1.0 - 0.5 / self.tau)
        tr = [k * v for v in tr]
        tn = sum(tr[a] * nrm[a] for a in range(3))
        out = torch.sqrt(sum((tr[a] - tn * nrm[a]) ** 2 for a in range(3)))
        wall = torch.as_tensor((self.lat.src == -1).any(axis=0), device=self.dev)
        return torch.where(wall, out, torch.full_like(out, float("nan")))


def _exact_adjoint(case, q, P):
    obj, n = q["objective"], case["steps"]
    dev = P.dev
    sites = torch.as_tensor(obj.sites, device=dev)
    target = torch.as_tensor(obj.target, device=dev)
    axis = [float(a) for a in obj.axis]
    tau = torch.tensor(q["tau"], dtype=torch.float64, device=dev, requires_grad=True)
    amps = torch.tensor(q["amps"], dtype=torch.float64, device=dev, requires_grad=True)

    def step(h, t):
        val = {k: (_wave_at(q["wave"], t) if io.kind == geometry.VELOCITY else 1.0) for k, io in enumerate(P.lat.iolets)}
        return P.stream(P.collide(h, tau), amps, val)[0]

    def cost(h):
        _, _, u = P.moments(h[:, sites])
        return ((sum(axis[a] * u[a] for a in range(3)) - target) ** 2).sum() / n

    states = [torch.zeros((19, P.n), dtype=torch.float64, device=dev)]
    with torch.no_grad():
        J = 0.0
        for t in range(n):
            states.append(step(states[-1], t))
            J += float(cost(states[-1]))
        _, rho, u = P.moments(states[-1])
    mu, dtau, damps = torch.zeros_like(states[0]), 0.0, torch.zeros_like(amps)
    for t in reversed(range(n)):
        h = states.pop()
        with torch.enable_grad():
            h = h.detach().requires_grad_(True)
            mu = mu + torch.autograd.grad(cost(h), h)[0]
            h = states[-1].detach().requires_grad_(True)
            g = torch.autograd.grad(step(h, t), (h, tau, amps), mu)
        mu, dtau, damps = g[0], dtau + float(g[1]), damps + g[2]
    return {"J": torch.tensor(J, dtype=torch.float64), "dtau": torch.tensor(dtau, dtype=torch.float64), "damps": damps,
            "rho": rho, "u": torch.stack(u)}


def exact(case, seed):
    lattice = _lattice(case)
    q = _inputs(case, seed, lattice)
    dev = _device()
    P = _Plain(lattice, q["tau"], dev)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, q, P)
    with torch.no_grad():
        amps = torch.as_tensor(q["amps"], device=dev)
        h = P.equilibrium(q["u0"])
        if case["precision"] != "fp64":                    # the start as it is stored: the inputs of the steps
            h = h.to({"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}[case["precision"]]).double()
        K = len(lattice.iolets)
        wk = {k: {"par": p, "rho": p[3], "ghost": p[3]} for k, p in enumerate(q.get("wk", []), 1)}
        series = {"flux": [], "u_max": [], "pressure": []}
        flux = {}
        for t in range(case["steps"]):
            val = {k: (_wave_at(q["wave"], t) if io.kind == geometry.VELOCITY else wk[k]["ghost"] if k in wk else 1.0)
                   for k, io in enumerate(lattice.iolets)}
            h, flux = P.stream(P.collide(h, q["tau"]), amps, val)
            for k, m in wk.items():
                rp, c, rd, rho_d = m["par"]
                out = -flux[k]
                if c > 0:
                    m["rho"] += (out - (m["rho"] - rho_d) / rd) / c
                    m["ghost"] = m["rho"] + rp * out
                else:
                    m["ghost"] = rho_d + (rp + rd) * out
            if case["kind"] == "monitor" and (t + 1) % case["every"] == 0:
                row = {"flux": [flux[k] for k in range(K)], "u_max": [0.0] * K, "pressure": [0.0] * K}
                for L in P.iolet:
                    x = torch.unique(L["x"])
                    _, rho, u = P.moments(h[:, x])
                    row["u_max"][L["k"]] = float(torch.sqrt(u[0] ** 2 + u[1] ** 2 + u[2] ** 2).max())
                    row["pressure"][L["k"]] = float(rho.mean()) / 3.0
                for key in series:
                    series[key].append(row[key])
        drho, rho, u = P.moments(h)
        if case["kind"] == "monitor":
            return {**{k: np.array(v) for k, v in series.items()}, "rho": rho, "u": torch.stack(u)}
        out = {"rho": rho, "u": torch.stack(u), "wss": P.wss(h)}
        if case["check"]:
            out["mass"] = float(P.n + drho.sum())
            out["flux"] = np.array([flux[k] for k in range(K)])
        return out
