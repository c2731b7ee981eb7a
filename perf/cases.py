"""Performance cases of the direct N-body library, through its public entry points.

`listed()` covers what programs do with the library: single force evaluations
(`Simulation.accel`), runs of the KDK leapfrog and of the fourth-order schemes
(`Simulation.step`, `get_state`, `get_accel`, `diagnostics`), the row share of
one GPU (`Simulation.accel_rows`) and ticks of the serving pool
(`serve.Batch`), in every precision mode, from 10^3 to 2^20 particles.
`draw()` gives more cases of the same ranges.
"""
import math

import numpy as np
import torch

import paper_1803_01190_gb300 as nb
from paper_1803_01190_gb300 import serve

#: Most pair interactions (N^2 per force evaluation) that a drawn case asks of each mode, a pass:
#: what the listed cases of that mode ask at most, on the slowest kernels.
_MOST = {"fp64": 2.0 ** 34, "f64e": 1.5 * 2.0 ** 34, "mixed": 2.0 ** 40, "fp32": 2.0 ** 38}

_FORCES = {"kdk": 1, "fr4": 3, "rk4": 4}  # force evaluations per step


def listed():
    return [
        # one evaluation of a small system: a call's own latency
        {"name": "accel fp64 1000", "do": "accel", "mode": "fp64", "n": 1000, "cloud": "plummer",
         "eps": 0.01, "host": False},
        # the small benchmark: Plummer sphere, 10 KDK steps, energies and momenta at the end
        {"name": "kdk fp64 4096", "do": "steps", "mode": "fp64", "n": 4096, "cloud": "plummer",
         "eps": 0.01, "scheme": "kdk", "dt": 1e-3, "steps": 10},
        # one evaluation of an ordinary system of odd size
        {"name": "accel fp64 20011", "do": "accel", "mode": "fp64", "n": 20011, "cloud": "disk",
         "eps": 0.02, "host": False},
        # the disk + halo benchmark in binary64: one step of a long run
        {"name": "kdk fp64 131072", "do": "steps", "mode": "fp64", "n": 131072, "cloud": "disk",
         "eps": 0.02, "scheme": "kdk", "dt": 5e-4, "steps": 1},
        # one GPU's share of a force sum split over eight
        {"name": "rows fp64 65536", "do": "rows", "mode": "fp64", "n": 65536, "rows": 8192,
         "cloud": "disk", "eps": 0.02},
        # a fourth-order step with binary64-class forces
        {"name": "fr4 f64e 65539", "do": "steps", "mode": "f64e", "n": 65539, "cloud": "disk",
         "eps": 0.02, "scheme": "fr4", "dt": 1.5e-3, "steps": 1},
        # a small system in the mixed mode, ten steps between outputs
        {"name": "kdk mixed 2048", "do": "steps", "mode": "mixed", "n": 2048, "cloud": "plummer",
         "eps": 0.01, "scheme": "kdk", "dt": 5e-4, "steps": 10},
        # one evaluation on host arrays, uneven masses, small softening (the precision sweep's)
        {"name": "accel mixed 16387 host", "do": "accel", "mode": "mixed", "n": 16387,
         "cloud": "uniform", "eps": 0.001, "host": True},
        # the disk + halo benchmark in the mixed mode
        {"name": "kdk mixed 131072", "do": "steps", "mode": "mixed", "n": 131072, "cloud": "disk",
         "eps": 0.02, "scheme": "kdk", "dt": 5e-4, "steps": 4},
        # and at its full size
        {"name": "kdk mixed 1048576", "do": "steps", "mode": "mixed", "n": 1048576,
         "cloud": "disk", "eps": 0.02, "scheme": "kdk", "dt": 5e-4, "steps": 1},
        # single precision (the paper's), classical Runge-Kutta
        {"name": "rk4 fp32 65536", "do": "steps", "mode": "fp32", "n": 65536, "cloud": "disk",
         "eps": 0.02, "scheme": "rk4", "dt": 2e-3, "steps": 2},
        # serving: a pool of simulations of uneven size, binary64 and mixed requests, four ticks
        {"name": "serve 12", "do": "serve", "sims": 12, "smallest": 1024, "largest": 32768,
         "fp64": 0.5, "ticks": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["accel", "accel", "steps", "steps", "steps", "rows", "serve"])
    if do == "serve":
        return {"do": "serve", "sims": rng.randint(2, 14), "smallest": 1024,
                "largest": _log(rng, 2048, 32768), "fp64": rng.choice([0.0, 0.5, 1.0]),
                "ticks": rng.randint(1, 4)}
    mode = rng.choice(["fp64", "fp64", "f64e", "mixed", "mixed", "fp32"])
    cloud = rng.choice(["plummer", "disk", "uniform"])
    eps = rng.choice([0.01, 0.02, 0.001])
    hi = {"fp64": 131072, "f64e": 131072, "mixed": 1048576, "fp32": 524288}[mode]
    c = {"do": do, "mode": mode, "n": _log(rng, 1000, hi), "cloud": cloud, "eps": eps}
    most = _MOST[mode]
    if do == "accel":
        c["host"] = rng.random() < 0.3
    elif do == "rows":
        c["rows"] = max(1, c["n"] // rng.choice([2, 4, 8]))
    else:
        c["scheme"] = rng.choice(["kdk", "kdk", "fr4", "rk4"])
        c["dt"] = rng.choice([5e-4, 1e-3, 2e-3])
        per = _FORCES[c["scheme"]] * float(c["n"]) ** 2
        while per > most:  # a size whose one step costs no more than the listed ones
            c["n"] = int(c["n"] * 0.8)
            per = _FORCES[c["scheme"]] * float(c["n"]) ** 2
        c["steps"] = max(1, min(rng.choice([1, 2, 10]), int(most / 4 / per)))
    return c


# ---------------------------------------------------------------- inputs
def _generator(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, dtype=torch.float64, device=g.device)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device=g.device)


def _directions(g, n):
    v = _normal(g, n, 3)
    return v / v.norm(dim=1, keepdim=True)


def _inverse(u, x, density):
    """Values with the given density over the grid x, from uniform u."""
    cdf = torch.cumsum((density[1:] + density[:-1]) * 0.5 * (x[1:] - x[:-1]), 0)
    cdf = torch.cat([torch.zeros_like(cdf[:1]), cdf]) / cdf[-1]
    k = torch.searchsorted(cdf, u).clamp(1, x.numel() - 1)
    t = (u - cdf[k - 1]) / (cdf[k] - cdf[k - 1]).clamp_min(1e-300)
    return x[k - 1] + t * (x[k] - x[k - 1])


def _plummer(g, n, a):
    """Plummer sphere of mass 1 and radius a (untruncated), isotropic velocities."""
    u = _uniform(g, n).clamp(1e-12, 1 - 1e-12)
    r = a / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)
    q = torch.linspace(0, 1, 4097, dtype=torch.float64, device=g.device)
    speed = _inverse(_uniform(g, n), q, q * q * (1 - q * q).clamp_min(0) ** 3.5)
    speed = speed * math.sqrt(2.0 / a) * (1 + (r / a) ** 2) ** -0.25
    return r[:, None] * _directions(g, n), speed[:, None] * _directions(g, n)


def _cloud(kind, n, seed):
    """(pos, vel, mass) on the GPU: `plummer` (equal masses), `disk` (exponential disk in a
    live halo, 1:1, equal masses) or `uniform` (unit ball, lognormal masses, at rest)."""
    g = _generator(seed)
    if kind == "plummer":
        pos, vel = _plummer(g, n, 1.0)
        mass = torch.full((n,), 1.0 / n, dtype=torch.float64, device=g.device)
    elif kind == "uniform":
        pos = _uniform(g, n)[:, None] ** (1.0 / 3.0) * _directions(g, n)
        vel = torch.zeros_like(pos)
        mass = torch.exp(0.5 * _normal(g, n))
        mass = mass / mass.sum()
    else:
        nd = n // 2
        x = torch.linspace(0, 5, 4097, dtype=torch.float64, device=g.device)
        R = _inverse(_uniform(g, nd), x, x * torch.exp(-x))
        phi = 2 * math.pi * _uniform(g, nd)
        z = 0.05 * torch.atanh((2 * _uniform(g, nd) - 1).clamp(-1 + 1e-12, 1 - 1e-12))
        inside = 1 - (1 + R) * torch.exp(-R) + R ** 3 / (R * R + 9) ** 1.5
        vc = torch.sqrt(inside / R.clamp_min(1e-3))
        e_r = torch.stack([torch.cos(phi), torch.sin(phi), torch.zeros_like(phi)], 1)
        e_p = torch.stack([-torch.sin(phi), torch.cos(phi), torch.zeros_like(phi)], 1)
        dpos = R[:, None] * e_r
        dpos[:, 2] = z
        dvel = vc[:, None] * e_p + 0.2 * vc[:, None] * _normal(g, nd, 3)
        hpos, hvel = _plummer(g, n - nd, 3.0)
        pos, vel = torch.cat([dpos, hpos]), torch.cat([dvel, hvel])
        mass = torch.full((n,), 2.0 / n, dtype=torch.float64, device=g.device)
    # a drift and an offset, so that the total momentum and angular momentum are not round-off
    vel = vel + torch.tensor([0.1, -0.05, 0.02], dtype=torch.float64, device=g.device)
    pos = pos + torch.tensor([0.02, 0.03, -0.01], dtype=torch.float64, device=g.device)
    return pos.contiguous(), vel.contiguous(), mass.contiguous()


def _pool(case, seed):
    """The simulations of a serving case: sizes log-uniform, two clouds, each its own state."""
    r = np.random.Generator(np.random.PCG64([int(seed) % (1 << 62), 77]))
    sims = []
    for k in range(case["sims"]):
        # sizes and modes are the case's, the same for every seed
        u = ((k * 0.6180339887498949) + 0.15) % 1.0
        n = int(round(math.exp(math.log(case["smallest"])
                               + u * math.log(case["largest"] / case["smallest"]))))
        kind = ("plummer", "disk")[k % 2]
        mode = "fp64" if ((k * 0.7548776662466927) % 1.0) < case["fp64"] else "mixed"
        sims.append({"n": n, "kind": kind, "mode": mode, "eps": 0.01 if kind == "plummer" else 0.02,
                     "seed": int(r.integers(1, 1 << 60))})
    return sims


# ---------------------------------------------------------------- the passes
def prepare(case, seed):
    if case["do"] == "serve":
        sims = _pool(case, seed)
        b = serve.Batch(capacity=sum(s["n"] + 64 for s in sims), max_sims=len(sims))
        for s in sims:
            pos, vel, mass = (t.cpu().numpy() for t in _cloud(s["kind"], s["n"], s["seed"]))
            s["slot"] = b.admit(pos, vel, mass, mode=s["mode"], eps=s["eps"], dt=5e-4)
        return {"case": case, "batch": b, "slots": [s["slot"] for s in sims]}
    pos, vel, mass = _cloud(case["cloud"], case["n"], seed)
    sim = nb.Simulation(case["n"], mode=case["mode"], eps=case["eps"])
    if case["do"] == "steps":
        sim.set_state(pos, vel, mass)
        return {"case": case, "sim": sim}
    if case.get("host"):
        pos, mass = pos.cpu().numpy(), mass.cpu().numpy()
    return {"case": case, "sim": sim, "pos": pos, "mass": mass}


def _rows(case):
    """The middle share of the rows."""
    return (case["n"] - case["rows"]) // 2, case["rows"]


def run(state):
    case = state["case"]
    if case["do"] == "accel":
        return state["sim"].accel(state["pos"], state["mass"])
    if case["do"] == "rows":
        return state["sim"].accel_rows(*_rows(case), state["pos"], state["mass"])
    if case["do"] == "serve":
        b = state["batch"]
        b.step(case["ticks"])
        return [(b.get_state(s)[:2], b.get_accel(s)) for s in state["slots"]]
    sim = state["sim"]
    sim.step(case["dt"], case["steps"], scheme=case["scheme"])
    pos, vel, _, _ = sim.get_state(on_device=True)
    if case["scheme"] == "rk4":  # its accelerations are not those of the state it ends in
        return pos, vel
    acc, pot = sim.get_accel(on_device=True)
    d = sim.diagnostics()
    return pos, vel, acc, pot, d["E"], d["P"], d["L"]


# ---------------------------------------------------------------- work and tolerances
def work(case):
    """Compulsory bytes (state in, results out, binary64 at the interface) and 20 flops per
    interaction, N^2 interactions per force evaluation."""
    if case["do"] == "serve":
        ns = [s["n"] for s in _pool(case, 0)]
        return {"bytes": float(sum(ns)) * 8 * (7 + 10) * case["ticks"],
                "flops": 20.0 * case["ticks"] * sum(float(n) * n for n in ns)}
    n = float(case["n"])
    if case["do"] == "accel":
        return {"bytes": n * 8 * 8, "flops": 20 * n * n}
    if case["do"] == "rows":
        return {"bytes": 8 * (4 * n + 4 * case["rows"]), "flops": 20 * n * case["rows"]}
    k = case["steps"] * _FORCES[case["scheme"]]
    return {"bytes": k * n * 8 * (7 + 6 + 4), "flops": 20 * n * n * k}


def tolerance(case):
    # about four times the largest relative error against `exact` seen for each mode: binary64
    # 2-5e-16 (1.1e-15 over a pool's simulations), f64e 1e-14 to 1e-13, mixed 5e-7 (2e-6 at
    # eps = 0.001, where single close pairs dominate), fp32 1e-6
    if case["do"] == "serve":
        rel = 2e-6 if case["fp64"] < 1 else 5e-15
    elif case["mode"] == "mixed":
        rel = 8e-6 if case["eps"] < 0.005 else 2e-6
    else:
        rel = {"fp64": 2e-15, "f64e": 4e-13, "fp32": 4e-6}[case["mode"]]
    return {"rel": rel, "max": 500 * rel}


# ---------------------------------------------------------------- the same in 64 bits
def _accel64(pos, mass, eps, i0=0, ni=None):
    """Accelerations and potentials in binary64, row blocks against all particles."""
    n = pos.shape[0]
    i1 = n if ni is None else i0 + ni
    acc, pot = [], []
    step = max(1, min(4096, (1 << 27) // n))
    cols = pos.t().contiguous()
    for a in range(i0, i1, step):
        b = min(i1, a + step)
        d = [cols[c][None, :] - cols[c][a:b, None] for c in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps
        r2[torch.arange(b - a), torch.arange(a, b)] = math.inf  # j == i
        y = r2.sqrt_().reciprocal_()
        my = y * mass
        pot.append(-my.sum(1))
        f = my.mul_(y).mul_(y)
        acc.append(torch.stack([(f * x).sum(1) for x in d], 1))
    return torch.cat(acc), torch.cat(pot)


def _diagnostics64(pos, vel, mass, pot):
    m = mass[:, None]
    E = float((0.5 * mass * (vel * vel).sum(1)).sum() + 0.5 * (mass * pot).sum())
    return E, (m * vel).sum(0).cpu().numpy(), (m * torch.linalg.cross(pos, vel)).sum(0).cpu().numpy()


def _kdk64(pos, vel, mass, eps, sizes):
    """KDK steps of the given sizes: (pos, vel, acc, pot)."""
    a, pot = _accel64(pos, mass, eps)
    for h in sizes:
        vt = vel + h * a
        pos = pos + 0.5 * h * (vt + vel)
        a, pot = _accel64(pos, mass, eps)
        vel = 0.5 * (vel + vt) + 0.5 * h * a
    return pos, vel, a, pot


def exact(case, seed):
    if case["do"] == "serve":
        out = []
        for s in _pool(case, seed):
            pos, vel, mass = _cloud(s["kind"], s["n"], s["seed"])
            # a simulation's first tick evaluates a(t0): one step fewer than ticks
            p, v, a, q = _kdk64(pos, vel, mass, s["eps"], [5e-4] * (case["ticks"] - 1))
            out.append(((p.cpu().numpy(), v.cpu().numpy()), (a.cpu().numpy(), q.cpu().numpy())))
        return out
    pairs = float(case["n"]) * case.get("rows", case["n"])
    if case["do"] == "steps":
        pairs *= _FORCES[case["scheme"]] * case["steps"] + 1
    if pairs > 7e10:
        return None
    pos, vel, mass = _cloud(case["cloud"], case["n"], seed)
    eps = case["eps"]
    if case["do"] in ("accel", "rows"):
        acc, pot = _accel64(pos, mass, eps, *(_rows(case) if case["do"] == "rows" else ()))
        return (acc.cpu().numpy(), pot.cpu().numpy()) if case.get("host") else (acc, pot)
    dt, steps = case["dt"], case["steps"]
    if case["scheme"] == "rk4":
        for _ in range(steps):
            a1 = _accel64(pos, mass, eps)[0]
            v2 = vel + 0.5 * dt * a1
            a2 = _accel64(pos + 0.5 * dt * vel, mass, eps)[0]
            v3 = vel + 0.5 * dt * a2
            a3 = _accel64(pos + 0.5 * dt * v2, mass, eps)[0]
            v4 = vel + dt * a3
            a4 = _accel64(pos + dt * v3, mass, eps)[0]
            pos = pos + dt / 6 * (vel + 2 * v2 + 2 * v3 + v4)
            vel = vel + dt / 6 * (a1 + 2 * a2 + 2 * a3 + a4)
        return pos, vel
    if case["scheme"] == "fr4":
        w1 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
        w0 = -(2.0 ** (1.0 / 3.0)) * w1
        sizes = [w1 * dt, w0 * dt, w1 * dt] * steps
    else:
        sizes = [dt] * steps
    pos, vel, acc, pot = _kdk64(pos, vel, mass, eps, sizes)
    return (pos, vel, acc, pot) + _diagnostics64(pos, vel, mass, pot)
