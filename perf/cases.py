"""The workloads whose speed this framework is judged by: what its users run, through its public entry points.

Three families, each over the sizes that the configurations, tests and benchmark of this repository use:

* boxes (``lb.Simulation``): the coupled fluctuating lattice Boltzmann + bead-spring chain step, one box.  A pass advances
  the box and takes the whole state out: populations (page-locked host memory, the C ABI's own layout) and beads.
* ensembles (``lb.Batch``): independent boxes advanced in lockstep, read out replica by replica.
* the chain side: the adjoint of the coupled step, Brownian dynamics with hydrodynamic interaction, and the FP64
  observables of a recorded trajectory.

The C ABI hands every result over as FP64.  Results of a context that computes in single precision are returned as FP32,
the type they were computed in.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0903_5067_gb300 import analysis, autograd, inputs, lb

PRECISION = {"f64": lb.LB_FP64, "f32": lb.LB_FP32, "bf16": lb.LB_BF16, "fp16": lb.LB_FP16}
STORED = {"f64": 8, "f32": 4, "bf16": 2, "fp16": 2}

# The two parameter sets of the repository: the configurations' fluid and chain, and the paper's production run (Sec. II E:
# two MD steps per LB step).
MODELS = {
    "config": dict(rho=1.0, eta=3.0, eta_b=3.0, kT=1.0, h=0.01, a=1.0, m=1.0, zeta=20.8, k_fene=30.0, R0=1.5, eps=1.0,
                   sigma=1.0),
    "paper": dict(rho=0.864, eta=0.864 * 2.8, eta_b=0.864 * 2.8, kT=1.2, h=0.02, a=1.0, m=1.0, zeta=20.8, k_fene=7.0,
                  R0=2.0, eps=1.0, sigma=1.0),
}
FLUID = ("rho", "eta", "eta_b", "kT", "h", "a")
CHAIN = ("m", "zeta", "k_fene", "R0", "eps", "sigma")

KS = [0.1 * 1.25 ** q for q in range(16)]  # the wave numbers of the structure factors


def listed():
    return [
        # The plain FP64 configuration: a small box, where launches and latency are all there is.
        dict(name="box_f64_L16_N8", kind="box", model="config", precision="f64", L=16, N=8, substeps=1, steps=200, upload=False,
             noise=True),
        # One box of the paper's production run: odd L, two MD steps per LB step.
        dict(name="box_f32_L25_N32_md2", kind="box", model="paper", precision="f32", L=25, N=32, substeps=2, steps=200,
             upload=False, noise=True),
        # The plain FP32 configuration: a box that stays in the L2 cache.
        dict(name="box_f32_L64_N64", kind="box", model="config", precision="f32", L=64, N=64, substeps=1, steps=200,
             upload=False, noise=True),
        # The headline workload: populations larger than the L2 cache.
        dict(name="box_f32_L128_N128", kind="box", model="config", precision="f32", L=128, N=128, substeps=1, steps=300,
             upload=False, noise=True),
        # The same box in 16-bit storage (the precision configuration).
        dict(name="box_bf16_L128_N128", kind="box", model="config", precision="bf16", L=128, N=128, substeps=1, steps=300,
             upload=False, noise=True),
        # The plain FP64 fluid that the single-precision results are checked against, from a given flow field and back.
        dict(name="fluid_f64_L72_upload", kind="box", model="config", precision="f64", L=72, N=0, substeps=1, steps=20,
             upload=True, noise=True),
        # The batching configuration: 64 boxes of five sizes and four chain lengths.
        dict(name="ensemble_c4", kind="ensemble", model="config", precision="f32", L=0, N=0, replicas=64, substeps=1, steps=240,
             frames=1),
        # The production ensemble of the paper's Table 1: 64 equal small boxes, beads read every 2 time units.
        dict(name="ensemble_L15_N32_md2", kind="ensemble", model="paper", precision="f32", L=15, N=32, replicas=64, substeps=2,
             steps=100, frames=4),
        # The differentiation configuration, through torch autograd.
        dict(name="adjoint_L32_N16", kind="adjoint", precision="f32", L=32, N=16, T=100, K=10),
        # Brownian dynamics of the paper's production chain, 64 chains.
        dict(name="bd_f32_64xN32", kind="bd", precision="f32", replicas=64, N=32, hi=True, steps=50),
        # Structure factors and hydrodynamic radius of a recorded run of the N = 128 chain.
        dict(name="structure_T1000_N128", kind="structure", T=1000, N=128, nk=16, nk_t=4, max_lag=100, stride=20),
        # Mean-square displacements and Rouse modes of the same run.
        dict(name="motion_T1000_N128", kind="motion", T=1000, N=128, max_lag=500),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _longest_chain(L):
    """The longest chain whose estimated 2 R_g fits the box (the rule of the batching configuration), at most 128."""
    return max(2, min(128, int((((L / 2.0) ** 2) * 6.5 / 0.97 ** 2) ** (1.0 / 1.176))))


def draw(rng):
    kind = rng.choice(["box", "box", "box", "ensemble", "ensemble", "adjoint", "bd", "structure", "motion"])
    if kind == "box":
        precision = rng.choice(["f32", "f32", "f32", "f64", "bf16", "fp16"])
        L = _log_int(rng, 8, 64 if precision == "f64" else 128)
        N = 0 if rng.random() < 0.2 else _log_int(rng, 2, _longest_chain(L))
        return dict(kind="box", model=rng.choice(["config", "paper"]), precision=precision, L=L, N=N,
                    substeps=rng.choice([1, 1, 2]) if N else 1, steps=rng.randint(10, 20) if precision == "f64" and L > 32
                    else rng.randint(40, 200), upload=rng.random() < 0.3, noise=rng.random() < 0.85)
    if kind == "ensemble":
        L = _log_int(rng, 8, 40)
        return dict(kind="ensemble", model=rng.choice(["config", "paper"]), precision=rng.choice(["f32", "f32", "f32", "f64"])
                    if L <= 16 else "f32", L=L, N=_log_int(rng, 2, min(64, _longest_chain(L))), replicas=_log_int(rng, 4, 64),
                    substeps=rng.choice([1, 2]), steps=rng.randint(20, 60), frames=rng.choice([1, 2]))
    if kind == "adjoint":
        L = _log_int(rng, 12, 40)
        return dict(kind="adjoint", precision="f32", L=L, N=_log_int(rng, 4, min(32, _longest_chain(L))),
                    T=rng.randint(40, 100), K=rng.randint(5, 15))
    if kind == "bd":
        precision = rng.choice(["f32", "f32", "f64"])
        return dict(kind="bd", precision=precision, replicas=_log_int(rng, 1, 160), N=_log_int(rng, 8, 74 if precision == "f32"
                    else 40), hi=rng.random() < 0.85, steps=rng.randint(10, 40))
    if kind == "structure":
        return dict(kind="structure", T=_log_int(rng, 100, 1000), N=_log_int(rng, 8, 128), nk=rng.randint(4, 16),
                    nk_t=rng.randint(1, 4), max_lag=rng.randint(10, 99), stride=rng.randint(5, 40))
    T = _log_int(rng, 200, 1600)
    return dict(kind="motion", T=T, N=_log_int(rng, 8, 128), max_lag=rng.randint(50, T // 2))


# --- inputs -----------------------------------------------------------------------------------------------------------
def _walk(N, L, seed):
    """A self-avoiding initial chain; another start where the walk gets stuck."""
    for again in range(50):
        try:
            return inputs.chain_walk(N, L=L, bond=0.97, seed=seed + 100003 * again, self_avoiding=True)
        except ValueError:
            continue
    raise ValueError("no self-avoiding walk")


def _pinned(n):
    return torch.empty(n, dtype=torch.float64, pin_memory=True)


def _flow(case, seed):
    """A flow field away from equilibrium: the rest state with 1 % perturbations."""
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12) * MODELS[case["model"]]["rho"]
    return w[:, None, None, None] * (1.0 + inputs.perturbation(case["L"], amplitude=1e-2, seed=seed))


def _ensemble(case, seed):
    """(L, N, seeds, initial chains) of the replicas: the batching configuration's mix, or equal boxes."""
    R = case["replicas"]
    if case["L"] == 0:
        return inputs.c4_ensemble(R, base_seed=100 + seed)
    seeds = [1000 * case["L"] + 7 * seed + r for r in range(R)]
    return [case["L"]] * R, [case["N"]] * R, seeds, [_walk(case["N"], case["L"], s) for s in seeds]


def _trajectory(case, seed):
    """A recorded run: a self-avoiding coil whose beads move about their places while its centre diffuses."""
    T, N = case["T"], case["N"]
    rng = np.random.default_rng(np.random.PCG64(seed))
    dev = np.empty((T, N, 3))
    dev[0] = 0.2 * rng.standard_normal((N, 3))
    kick = 0.2 * math.sqrt(1 - 0.98 ** 2) * rng.standard_normal((T, N, 3))
    for t in range(1, T):
        dev[t] = 0.98 * dev[t - 1] + kick[t]
    centre = np.cumsum(0.02 * rng.standard_normal((T, 1, 3)), axis=0)
    return torch.tensor(_walk(N, 32 if N <= 128 else 64, seed) + centre + dev, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "box":
        p = MODELS[case["model"]]
        L, N = case["L"], case["N"]
        sim = lb.Simulation(L=L, seed=seed, precision=PRECISION[case["precision"]], **{k: p[k] for k in FLUID})
        if N:
            sim.add_chain(N, x0=_walk(N, L, seed), **{k: p[k] for k in CHAIN})
        sim.set_md_substeps(case["substeps"])
        if not case["noise"]:
            sim.set_options(noise_fluid=0, noise_beads=0)
        state = dict(case=case, sim=sim, out=_pinned(19 * L ** 3))
        if case["upload"]:
            state["flow"] = _pinned(19 * L ** 3)
            state["flow"].numpy()[:] = _flow(case, seed).reshape(-1)
        sim.step(0)  # the box is on the device
        sim.sync()
        return state
    if kind == "ensemble":
        Ls, Ns, seeds, X = _ensemble(case, seed)
        b = lb.Batch(Ls, Ns, seeds, X, precision=PRECISION[case["precision"]], md_substeps=case["substeps"],
                     **MODELS[case["model"]])
        b.sync()
        return dict(case=case, batch=b, L=Ls, N=Ns, out=_pinned(19 * sum(L ** 3 for L in Ls)))
    if kind == "adjoint":
        x0 = torch.tensor(_walk(case["N"], case["L"], seed), dtype=torch.float32, device="cuda", requires_grad=True)
        zeta = torch.tensor(20.8, dtype=torch.float32, device="cuda", requires_grad=True)
        return dict(case=case, x0=x0, zeta=zeta,
                    params=dict(L=case["L"], seed=seed, precision=PRECISION[case["precision"]]))
    if kind == "bd":
        X = np.stack([_walk(case["N"], 1000, 100 * seed + r) for r in range(case["replicas"])])
        return dict(case=case, bd=lb.BD(X, precision=PRECISION[case["precision"]], seed=seed, hi=case["hi"]))
    return dict(case=case, traj=_trajectory(case, seed))


# --- one pass ---------------------------------------------------------------------------------------------------------
def _typed(case, a):
    """A result as the type it was computed in."""
    t = torch.from_numpy(a) if isinstance(a, np.ndarray) else a
    return t if case["precision"] == "f64" else t.to(torch.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "box":
        sim, L = state["sim"], case["L"]
        if case["upload"]:
            lb.lb_set_populations(sim.ctx, state["flow"].numpy())
        sim.step(case["steps"])
        lb.lb_get_populations(sim.ctx, state["out"].numpy())
        out = {"n": _typed(case, state["out"].view(19, L, L, L))}
        if case["N"]:
            x, v = sim.beads()
            out["x"], out["v"] = _typed(case, x), _typed(case, v)
        return out
    if kind == "ensemble":
        b = state["batch"]
        frames = []
        for _ in range(case["frames"]):
            b.step(case["steps"])
            read = [b.beads(r) for r in range(len(state["L"]))]
            frames.append([_typed(case, np.concatenate([w[q] for w in read])) for q in (0, 1)])
        at, n = 0, state["out"].numpy()
        for r, L in enumerate(state["L"]):
            lb.lb_batch_get_populations(b.b, r, n[at:at + 19 * L ** 3])
            at += 19 * L ** 3
        return {"n": _typed(case, state["out"]), "x": torch.stack([f[0] for f in frames]),
                "v": torch.stack([f[1] for f in frames])}
    if kind == "adjoint":
        O = autograd.chain_displacement(state["x0"], state["zeta"], state["params"], T=case["T"], K=case["K"])
        gx, gz = torch.autograd.grad(O, (state["x0"], state["zeta"]))
        return {"O": O.detach(), "gx": gx, "gz": gz}
    if kind == "bd":
        state["bd"].step(case["steps"])
        return {"x": _typed(case, state["bd"].beads())}
    traj = state["traj"]
    if kind == "structure":
        return {"S": analysis.static_sk(traj, KS[:case["nk"]]),
                "St": analysis.dynamic_sk(traj, KS[:case["nk_t"]], case["max_lag"], origin_stride=case["stride"]),
                "inv_R": analysis.inverse_radius(traj)}
    g1, g2, g3 = analysis.msd(traj, case["max_lag"])
    X = analysis.rouse_modes(traj)
    c, _ = analysis.rouse_correlation(X, case["max_lag"])
    return {"g1": g1, "g2": g2, "g3": g3, "X": X, "c": c}


# --- what one pass cannot do without ----------------------------------------------------------------------------------
NODE_FLOPS = 350  # moments, relaxation, back-transform and 15 Gaussians of one node update


def work(case):
    kind = case["kind"]
    if kind in ("box", "ensemble"):
        s = STORED[case["precision"]]
        Ls, Ns = ([case["L"]], [case["N"]]) if kind == "box" else _shapes(case)
        nodes = sum(L ** 3 for L in Ls)
        steps = case["steps"] * case.get("frames", 1)
        io = 19 * 8 * nodes * (2 if case.get("upload") else 1) + 48 * sum(Ns) * case.get("frames", 1)
        pairs = sum(N * N for N in Ns) * case["substeps"]
        return {"bytes": 38 * s * nodes * steps + io, "flops": (NODE_FLOPS * nodes + 30 * pairs) * steps}
    if kind == "adjoint":  # forward, recomputation and reverse sweep (which reads state and adjoint, and writes the adjoint)
        nodes, T = case["L"] ** 3, case["T"]
        return {"bytes": (38 + 38 + 57) * 4 * nodes * T, "flops": 3 * NODE_FLOPS * nodes * T}
    if kind == "bd":  # 62 products with the 3N x 3N mobility and its 3N x 3N entries, per chain and step
        n = 3 * case["N"]
        return {"bytes": 2 * 8 * n * case["replicas"], "flops": (62 * 2 * n * n + 10 * n * n if case["hi"] else 10 * n * n)
                * case["replicas"] * case["steps"]}
    T, N = case["T"], case["N"]
    if kind == "structure":  # 20 operations for each sine over its argument
        static = T * N * (N - 1) // 2 * case["nk"]
        pairs_t = sum((T - lag + case["stride"] - 1) // case["stride"] for lag in range(case["max_lag"] + 1) if lag < T) * N * N
        return {"bytes": 24 * T * N, "flops": 20 * (static + pairs_t * case["nk_t"]) + 15 * T * N * N}
    lags, P = case["max_lag"] + 1, N - 1
    return {"bytes": 24 * T * N + 2 * 24 * T * P + 8 * lags * (3 + P),
            "flops": 6 * T * N * P + sum(T - lag for lag in range(lags) if lag < T) * (60 + 6 * P)}


def _shapes(case):
    if case["L"]:
        return [case["L"]] * case["replicas"], [case["N"]] * case["replicas"]
    Ls, Ns, _, _ = inputs.c4_ensemble(case["replicas"])
    return Ls, Ns


# --- the same in plain torch, in 64 bits ------------------------------------------------------------------------------
VELOCITIES = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
              (0, -1, 1)]
M32 = 0xFFFFFFFF


def _philox(step, index, call, k0, k1):
    """Philox4x32-10 of the counters (step, index, call, 0): four int64 tensors of 32-bit words."""
    c = [torch.full_like(index, step & M32), index, torch.full_like(index, call), torch.zeros_like(index)]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _polar(u0, u1):
    r, th = torch.sqrt(-2.0 * torch.log(u0)), 2.0 * math.pi * (u1 - 0.5)
    return r * torch.cos(th), r * torch.sin(th)


def _bead_noise(step, N, k0, k1, device):
    """Three standard normals for each of N beads."""
    w = [((x >> 9).double() + 0.5) * 2.0 ** -23 for x in _philox(step, torch.arange(N, device=device), 0, k0, k1)]
    g0, g1 = _polar(w[0], w[1])
    return torch.stack([g0, g1, _polar(w[2], w[3])[0]], dim=1)


def _chain_forces(x, p, box=None):
    """FENE on bonds and WCA between all beads; x: (..., N, 3)."""
    N = x.shape[-2]
    d = x.unsqueeze(-2) - x.unsqueeze(-3)
    if box:
        d = d - box * torch.round(d.detach() / box)
    i = torch.arange(N, device=x.device)
    eye, bond = (i[:, None] == i[None]), (i[:, None] - i[None]).abs() == 1
    r2 = (d * d).sum(-1) + eye.double()
    s6 = (p["sigma"] ** 2 / r2) ** 3
    wca = torch.where((r2 < 2.0 ** (1 / 3) * p["sigma"] ** 2) & ~eye, 24 * p["eps"] / r2 * (2 * s6 * s6 - s6),
                      torch.zeros_like(r2))
    fene = torch.where(bond, -p["k_fene"] / (1 - torch.where(bond, r2, torch.zeros_like(r2)) / p["R0"] ** 2),
                       torch.zeros_like(r2))
    return ((wca + fene).unsqueeze(-1) * d).sum(-2)


class _Box:
    """One box and its chain in FP64; differentiable with respect to the initial positions and the friction."""

    def __init__(self, p, L, seed, replica=0, noise=True, substeps=1, n=None, x0=None, zeta=None, device="cuda"):
        self.p, self.L, self.nsub, self.noise, self.dev = p, L, substeps, noise, device
        self.zeta = p["zeta"] if zeta is None else zeta
        c = torch.tensor(VELOCITIES, dtype=torch.float64, device=device)
        x, y, z = c.T
        s = (c * c).sum(1)
        o = torch.ones_like(s)
        self.E = torch.stack([o, x, y, z, s - 1, 3 * x * x - s, y * y - z * z, x * y, y * z, x * z, (3 * s - 5) * x,
                              (3 * s - 5) * y, (3 * s - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y,
                              (x * x - y * y) * z, 3 * s * s - 6 * s + 1, (2 * s - 3) * (3 * x * x - s),
                              (2 * s - 3) * (y * y - z * z)])
        w = torch.tensor([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, dtype=torch.float64, device=device)
        b = (self.E ** 2) @ w
        self.back = (self.E * w[None] / b[:, None]).T.contiguous()
        nu, nub = (p[k] * p["h"] / (p["rho"] * p["a"] ** 2) for k in ("eta", "eta_b"))
        self.gs, self.gb = 1 - 2 / (6 * nu + 1), 1 - 2 / (9 * nub + 1)
        g = torch.zeros(19, dtype=torch.float64, device=device)
        g[4], g[5:10] = self.gb, self.gs
        self.g = g
        self.phi = torch.sqrt(3 * p["kT"] * p["h"] ** 2 / p["a"] ** 5 * b * (1 - g * g))
        self.key = (seed & M32, replica << 8)
        rest = (w * p["rho"])[:, None].expand(19, L ** 3)
        self.n = rest.clone() if n is None else torch.tensor(np.asarray(n), device=device).reshape(19, -1)
        self.N = 0 if x0 is None else x0.shape[0]
        self.k = 0
        if self.N:
            self.x = x0 if isinstance(x0, torch.Tensor) else torch.tensor(x0, device=device)
            self.v = torch.zeros_like(self.x)
            self.F = _chain_forces(self.x, p, L * p["a"])

    def _stress(self, rho, j, dJ):
        """Moment increments 1..9 of the force that adds momentum dJ (3, ...)."""
        U = (j + 0.5 * dJ) / rho
        cs = 0.5 * (1 + self.gs)
        diag = ((1 + self.gb) / 3 - 2 / 3 * cs) * (U * dJ).sum(0)
        P = [2 * cs * U[q] * dJ[q] + diag for q in range(3)]
        off = [cs * (U[q] * dJ[r] + U[r] * dJ[q]) for q, r in ((0, 1), (1, 2), (0, 2))]
        return torch.stack([dJ[0], dJ[1], dJ[2], P[0] + P[1] + P[2], 2 * P[0] - P[1] - P[2], P[1] - P[2], *off])

    def _beads(self, m):
        """The bead steps against the post-stream fluid m; the moment increments at the nodes they push."""
        p, L = self.p, self.L
        h = p["h"] / self.nsub
        nodes, push = [], []
        for sub in range(self.nsub):
            vh = self.v + h * self.F / (2 * p["m"])
            self.x = self.x + h * vh
            s = self.x / p["a"]
            cell = torch.floor(s.detach())
            f, cell = s - cell, cell.long()
            u = torch.zeros_like(self.x)
            corners = []
            for c in range(8):
                d = torch.tensor([c & 1, c >> 1 & 1, c >> 2 & 1], device=self.dev)
                w = torch.where(d.bool(), f, 1 - f).prod(1)
                q = (cell + d) % L
                node = q[:, 0] + L * (q[:, 1] + L * q[:, 2])
                u = u + w[:, None] * (m[1:4, node] / m[0, node]).T * (p["a"] / p["h"])
                corners.append((node, w))
            Fc = -self.zeta * (vh - u)
            if self.noise:
                g = _bead_noise(self.k * self.nsub + sub, self.N, self.key[0], 1 | self.key[1], self.dev)
                amp = 2 * p["kT"] * self.zeta / h
                Fc = Fc + (torch.sqrt(amp) if isinstance(amp, torch.Tensor) else math.sqrt(amp)) * g
            self.F = _chain_forces(self.x, p, L * p["a"]) + Fc
            self.v = vh + h * self.F / (2 * p["m"])
            for node, w in corners:
                nodes.append(node)
                push.append(-w[:, None] * Fc / self.nsub / p["a"] ** 3 * p["h"] ** 2 / p["a"])
        at, back = torch.unique(torch.cat(nodes), return_inverse=True)
        dJ = torch.zeros(at.numel(), 3, dtype=torch.float64, device=self.dev).index_add(0, back, torch.cat(push)).T
        return at, self._stress(m[0, at], m[1:4, at], dJ)

    def step(self):
        p, L = self.p, self.L
        n = self.n.view(19, L, L, L)
        n = torch.stack([torch.roll(n[i], shifts=(c[2], c[1], c[0]), dims=(0, 1, 2)) for i, c in enumerate(VELOCITIES)])
        m = self.E @ n.view(19, -1)
        rho, j = m[0], m[1:4]
        q = j * j / rho
        eq = [q[0] + q[1] + q[2], 2 * q[0] - q[1] - q[2], q[1] - q[2], j[0] * j[1] / rho, j[1] * j[2] / rho, j[0] * j[2] / rho]
        g = self.g[4:10, None]
        rest = list(g * m[4:10] + (1 - g) * torch.stack(eq)) + [torch.zeros_like(rho)] * 9
        if self.noise and p["kT"] > 0:
            index, sr = torch.arange(L ** 3, device=self.dev), torch.sqrt(rho)
            for call in range(2):
                for w, word in enumerate(_philox(self.k, index, call, *self.key)):
                    pair = _polar(((word >> 11).double() + 0.5) * 2.0 ** -21, ((word & 0x7FF).double() + 0.5) * 2.0 ** -11)
                    for half in range(2):
                        mode = 4 + 2 * (4 * call + w) + half
                        if mode < 19:
                            rest[mode - 4] = rest[mode - 4] + self.phi[mode] * sr * pair[half]
        post = self.back @ torch.cat([m[:4], torch.stack(rest)])
        if self.N:
            at, dm = self._beads(m)
            post = post.index_add(1, at, self.back[:, 1:10] @ dm)
        self.n = post
        self.k += 1


def _bd(case, seed):
    """Ito-Euler with the regularised Rotne-Prager-Yamakawa mobility and the Chebyshev square root, all chains at once."""
    N, R, dev = case["N"], case["replicas"], "cuda"
    n = 3 * N
    p = dict(kT=1.2, k_fene=7.0, R0=2.0, eps=1.0, sigma=1.0)
    eta = 0.864 * 2.8
    zeta = 1.0 / (1.0 / 20.8 + 1.0 / (25.0 * eta))
    dt, a = 0.005 * zeta / (4.0 * 7.0), zeta / (6 * math.pi * eta)
    x = torch.tensor(np.stack([_walk(N, 1000, 100 * seed + r) for r in range(R)]), device=dev)
    eye3, eye = torch.eye(3, dtype=torch.float64, device=dev), torch.eye(N, dtype=torch.bool, device=dev)
    start = torch.full((R, n, 1), 1 / math.sqrt(n), dtype=torch.float64, device=dev)
    K = 21
    theta = math.pi * (torch.arange(K, dtype=torch.float64, device=dev) + 0.5) / K
    for step in range(case["steps"]):
        F = _chain_forces(x, p)
        W = torch.stack([_bead_noise(step, N, seed & M32, 3 | r << 8, dev) for r in range(R)]).reshape(R, n, 1)
        d = x.unsqueeze(2) - x.unsqueeze(1)
        r2 = (d * d).sum(-1) + eye
        r = torch.sqrt(r2)
        far = r >= 2 * a
        ci = torch.where(far, (1 + 2 * a * a / r2 / 3) / (8 * math.pi * eta * r), (1 - 9 * r / a / 32) / (6 * math.pi * eta * a))
        cr = torch.where(far, (1 - 2 * a * a / r2) / (8 * math.pi * eta * r), 3 * r / a / 32 / (6 * math.pi * eta * a))
        blk = ci[..., None, None] * eye3 + (cr / r2)[..., None, None] * d.unsqueeze(-1) * d.unsqueeze(-2)
        if not case["hi"]:
            blk = torch.zeros_like(blk)
        blk = torch.where(eye[None, :, :, None, None], eye3 / zeta, blk)
        M = blk.permute(0, 1, 3, 2, 4).reshape(R, n, n)
        if case["hi"]:
            D = p["kT"] * M

            def largest(A):
                v = start
                for _ in range(20):
                    v = A @ v
                    v = v / v.norm(dim=1, keepdim=True)
                return (v * (A @ v)).sum(1, keepdim=True)

            top = 1.05 * largest(D)
            low = 0.5 * (top - largest(top * torch.eye(n, dtype=torch.float64, device=dev) - D))
            low = torch.maximum(low, top / 1000)
            f = torch.sqrt(0.5 * (top + low) + 0.5 * (top - low) * torch.cos(theta))  # (R, 1, K)
            c = [(1 if k == 0 else 2) / K * (f * torch.cos(k * theta)).sum(2, keepdim=True) for k in range(K)]
            A = 2 / (top - low) * D - (top + low) / (top - low) * torch.eye(n, dtype=torch.float64, device=dev)
            t0, t1 = W, A @ W
            y = c[0] * t0 + c[1] * t1
            for k in range(2, K):
                t0, t1 = t1, 2 * (A @ t1) - t0
                y = y + c[k] * t1
        else:
            y = math.sqrt(p["kT"] / zeta) * W
        x = x + (dt * (M @ F.reshape(R, n, 1)) + math.sqrt(2 * dt) * y).reshape(R, N, 3)
    return x


def _sinc(k, r):
    x = k * r
    return torch.where(x == 0, torch.ones_like(x), torch.sin(x) / torch.where(x == 0, torch.ones_like(x), x))


def _structure(case, seed):
    traj = _trajectory(case, seed)
    T, N = case["T"], case["N"]
    off = ~torch.eye(N, dtype=torch.bool, device=traj.device)
    S, inv = np.zeros(case["nk"]), 0.0
    for t in range(0, T, 50):
        r = (traj[t:t + 50, :, None] - traj[t:t + 50, None]).norm(dim=-1)
        S += np.array([_sinc(k, r).sum().item() for k in KS[:case["nk"]]])
        inv += (1 / r[:, off]).sum().item()
    St = np.zeros((case["nk_t"], case["max_lag"] + 1))
    for lag in range(min(case["max_lag"] + 1, T)):
        a = traj[0:T - lag:case["stride"]]
        r = (traj[lag::case["stride"]][:a.shape[0], :, None] - a[:, None]).norm(dim=-1)
        St[:, lag] = [_sinc(k, r).sum().item() / (N * a.shape[0]) for k in KS[:case["nk_t"]]]
    return {"S": S / (N * T), "St": St, "inv_R": inv / (N * N * T)}


def _motion(case, seed):
    traj = _trajectory(case, seed)
    T, N, lags = case["T"], case["N"], case["max_lag"] + 1
    cm = traj.mean(1)
    inner = traj[:, [(N - 1) // 2, N // 2]]
    g = np.zeros((3, lags))
    p, q = torch.arange(1, N, dtype=torch.float64, device=traj.device), torch.arange(N, dtype=torch.float64, device=traj.device)
    X = torch.einsum("tnc,pn->tpc", traj, torch.cos(math.pi / N * p[:, None] * (q[None] + 0.5))) / N
    c = np.zeros((N - 1, lags))
    for lag in range(min(lags, T)):
        d, dc = inner[lag:] - inner[:T - lag], (cm[lag:] - cm[:T - lag])[:, None]
        g[:, lag] = [(d * d).sum(-1).mean().item(), ((d - dc) ** 2).sum(-1).mean().item(), (dc * dc).sum(-1).mean().item()]
        c[:, lag] = (X[lag:] * X[:T - lag]).sum(-1).mean(0).cpu().numpy()
    return {"g1": g[0], "g2": g[1], "g3": g[2], "X": X, "c": c}


def exact(case, seed):
    kind = case["kind"]
    if kind == "box":
        L, N = case["L"], case["N"]
        box = _Box(MODELS[case["model"]], L, seed, noise=case["noise"], substeps=case["substeps"],
                   n=_flow(case, seed) if case["upload"] else None, x0=_walk(N, L, seed) if N else None)
        with torch.no_grad():
            for _ in range(case["steps"]):
                box.step()
        out = {"n": box.n.view(19, L, L, L)}
        return {**out, "x": box.x, "v": box.v} if N else out
    if kind == "ensemble":
        Ls, Ns, seeds, X = _ensemble(case, seed)
        if sum(L ** 3 for L in Ls) * case["steps"] * case["frames"] > 2e8 or len(Ls) * case["steps"] * case["frames"] > 3000:
            return None  # minutes in plain torch
        boxes = [_Box(MODELS[case["model"]], L, s, replica=r, substeps=case["substeps"], x0=X[r])
                 for r, (L, s) in enumerate(zip(Ls, seeds))]
        xs, vs = [], []
        with torch.no_grad():
            for _ in range(case["frames"]):
                for box in boxes:
                    for _ in range(case["steps"]):
                        box.step()
                xs.append(torch.cat([box.x for box in boxes]))
                vs.append(torch.cat([box.v for box in boxes]))
        return {"n": torch.cat([box.n.reshape(-1) for box in boxes]), "x": torch.stack(xs), "v": torch.stack(vs)}
    if kind == "adjoint":
        x0 = torch.tensor(_walk(case["N"], case["L"], seed), dtype=torch.float32, device="cuda").double().requires_grad_()
        zeta = torch.tensor(float(np.float32(20.8)), dtype=torch.float64, device="cuda", requires_grad=True)
        box = _Box(MODELS["config"], case["L"], seed, x0=x0, zeta=zeta)
        for _ in range(case["T"]):
            box.step()
        O = ((box.x - x0.detach()) ** 2).sum()
        return dict(zip(("O", "gx", "gz"), (O.detach(), *_displacement_gradients(box, x0, zeta))))
    if kind == "bd":
        return {"x": _bd(case, seed)}
    return _structure(case, seed) if kind == "structure" else _motion(case, seed)


def _displacement_gradients(box, x0, zeta):
    return torch.autograd.grad(((box.x - x0) ** 2).sum(), (x0, zeta))
