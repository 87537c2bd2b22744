"""The work that users of this package have it do, as cases that can be timed and compared.

Every case goes through the public entry points (``NBody``, ``accel_static``,
``autograd.trajectory``) on the seeded Solar-System-shaped models of
``inputs``.  A case's ``kind`` says which:

* ``step``   -- integrate: ``NBody.step``, then the state and the acceleration.
* ``grad``   -- dL/d(r0, v0, m) of a loss on the final state, ``NBody.grad``.
* ``train``  -- one optimisation iteration: trajectory forward and backward
  through ``torch.autograd``.
* ``energy`` -- the accuracy check of a run, ``NBody.energy``.
* ``static`` -- Eq. 1 without device allocation, ``accel_static``.

Moons faster than the step are chaotic under plain Verlet (any two roundings
part within a few steps), so integrations raise the drawn moon radii to
omega dt <= 0.5; only close-encounter handling, which resolves such moons,
takes them as drawn.

The mixed path's forces are FP32-accurate by design (its documented gate is
2e-6), so what depends on one force evaluation (accelerations), on their sum
over a short run (velocities) or on their derivative (gradients) is returned
as float32, as a user of that path stores it; positions, which that path
carries in FP64, come as float64.
"""
import math

import numpy as np
import torch

from paper_2112_15079_gb300 import autograd, inputs, nbody

RESOLVED = 0.5  # largest omega dt of a moon, where moons are resolved
CLOSE = (0.5, 0.05)  # close-encounter thresholds (theta_c, theta_s) of the repository's benchmark


def listed():
    return [
        # The Sun and 30 major bodies, the smallest model: launch and exchange latency are all there is.
        {"name": "steps_fp64_31", "kind": "step", "n": 31, "precision": "fp64", "steps": 100},
        # A reduced belt, odd size: a few hundred bodies still fit one launch, latency and FP64 chains.
        {"name": "steps_fp64_521", "kind": "step", "n": 521, "precision": "fp64", "steps": 20},
        # The paper's production model in full precision: the benchmark's FP64 headline.
        {"name": "steps_fp64_10425", "kind": "step", "n": 10425, "precision": "fp64", "steps": 10},
        # The same model in mixed precision, the benchmark's mixed headline: a day between snapshots.
        {"name": "steps_mixed_10425", "kind": "step", "n": 10425, "precision": "mixed", "steps": 10},
        # A denser belt, the middle of the benchmark's sweep.
        {"name": "steps_mixed_65536", "kind": "step", "n": 65536, "precision": "mixed", "steps": 4},
        # The largest model of the benchmark: one step, as a run that writes every snapshot takes it.
        {"name": "steps_mixed_1048576", "kind": "step", "n": 1048576, "precision": "mixed", "steps": 1},
        # An ensemble of independent systems of uneven size in one context.
        {"name": "ensemble_mixed_64", "kind": "step", "systems": 64, "lo": 1000, "hi": 20000, "precision": "mixed",
         "steps": 1},
        # Sensitivities of the production model: mixed precision, checkpoints inside the run.
        {"name": "grad_mixed_10425", "kind": "grad", "n": 10425, "precision": "mixed", "steps": 20, "ckpt": 8},
        # One iteration of fitting initial conditions in full precision, through torch.autograd.
        {"name": "train_fp64_2131", "kind": "train", "n": 2131, "precision": "fp64", "steps": 20, "ckpt": 0},
        # The paper's accuracy criterion, evaluated along a run.
        {"name": "energy_fp64_10425", "kind": "energy", "n": 10425, "precision": "fp64"},
        # A host that may not allocate: accelerations of the production model.
        {"name": "static_fp64_10425", "kind": "static", "n": 10425},
        # The production model with its fast moons resolved by close-encounter handling.
        {"name": "close_mixed_10425", "kind": "step", "n": 10425, "precision": "mixed", "steps": 5, "close": True},
    ]


def _size(rng, lo, hi):
    """Log-uniform in [lo, hi], mostly not a round number."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["fp64", "mixed", "integrator", "ensemble", "grad", "train", "energy", "static", "close"],
                       [4, 4, 2, 2, 2, 1, 1, 1, 1])[0]
    precision = rng.choice(["fp64", "mixed"])
    if kind in ("fp64", "mixed"):
        # up to one step of 131,072 (FP64) or 1,048,576 (mixed) bodies, down to many steps of a small model
        n = _size(rng, 31, 131072 if kind == "fp64" else 1048576)
        budget = 1.2e9 if kind == "fp64" else 1.2e10  # ordered pairs per call, for the smaller models
        # (a moon's orbit carries a mixed force error on as its phase, which grows with the square of the time)
        most = 200 if kind == "fp64" else 10
        return {"kind": "step", "n": n, "precision": kind, "steps": max(1, min(most, int(budget / n**2)))}
    if kind == "integrator":
        n = _size(rng, 31, 20000)
        return {"kind": "step", "n": n, "precision": precision, "steps": max(1, min(10, int(5e8 / n**2))),
                "integrator": rng.choice(["leapfrog", "rk4"])}
    if kind == "ensemble":
        lo = _size(rng, 40, 2000)
        return {"kind": "step", "systems": _size(rng, 2, 64), "lo": lo,
                "hi": min(20000, lo * rng.randint(2, 10)) if precision == "mixed" else 2 * lo,
                "precision": precision, "steps": 1}
    if kind in ("grad", "train"):
        n = _size(rng, 64, 10425 if kind == "grad" else 4096)
        return {"kind": kind, "n": n, "precision": precision, "steps": max(1, min(40, int(2e9 / n**2))),
                "ckpt": rng.choice([0, 3, 16])}
    if kind == "close":
        return {"kind": "step", "n": _size(rng, 131, 10425), "precision": precision, "steps": rng.randint(1, 8),
                "close": True}
    case = {"kind": kind, "n": _size(rng, 31, 65536)}
    return dict(case, precision="fp64") if kind == "energy" else case


def _systems(case, seed):
    base = inputs.BASE_SEED + 1000 * int(seed)
    omega = None if case.get("close") else RESOLVED
    if "systems" not in case:
        return [_draw_system(case["n"], base, omega)]
    sizes = np.random.default_rng([case["lo"], case["hi"]]).integers(case["lo"], case["hi"] + 1, case["systems"])
    return [_draw_system(int(k), base + i, omega) for i, k in enumerate(sizes)]


def _draw_system(n, seed, omega):
    for s in range(seed, seed + 100000, 1000):  # (a draw without a heavy planet has no hosts for its moons)
        try:
            return inputs.solar_system(n, s + 1, moon_omega_dt_max=omega)
        except ValueError:
            continue
    raise ValueError("no usable seed")


def _loss(case, seed, s):
    """dL/dr_T-like vectors of a loss on a seeded subset of the bodies: (indices, targets)."""
    rng = np.random.default_rng(seed + 17)
    idx = np.sort(rng.choice(np.arange(1, s.n), size=min(64, s.n - 1), replace=False))
    return idx, s.r[:, idx] + rng.normal(0.0, 1e-2, size=(3, len(idx)))


def prepare(case, seed):
    systems = _systems(case, seed)
    s = systems[0]
    dev = torch.device("cuda")
    state = {"case": case}
    if case["kind"] == "static":
        state.update(r=torch.tensor(s.r, device=dev), m=torch.tensor(s.m, device=dev), G=s.G)
        return state
    if case["kind"] == "train":
        idx, target = _loss(case, seed, s)
        state.update(r=torch.tensor(s.r, device=dev, requires_grad=True),
                     v=torch.tensor(s.v, device=dev, requires_grad=True),
                     m=torch.tensor(s.m, device=dev, requires_grad=True), G=s.G, dt=s.dt,
                     idx=torch.tensor(idx, device=dev), target=torch.tensor(target, device=dev))
        return state
    off, r, v, m = inputs.concat(systems)
    kw = dict(close_omega_dt=CLOSE[0], substep_omega_dt=CLOSE[1]) if case.get("close") else {}
    state["sim"] = nbody.NBody(r, v, m, off, G=s.G, dt=s.dt, precision=case["precision"],
                               ckpt_every=case.get("ckpt", 0), integrator=case.get("integrator", "verlet"), **kw)
    if case["kind"] == "grad":
        idx, target = _loss(case, seed, s)
        dr = np.zeros((3, s.n))
        dr[:, idx] = 2.0 * (s.r[:, idx] - target)
        state["dr"] = torch.tensor(dr, device=dev)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    kept = torch.float32 if case.get("precision") == "mixed" else torch.float64
    if kind == "static":
        return nbody.accel_static(state["r"], state["m"], state["G"])
    if kind == "train":
        rt, vt = autograd.trajectory(state["r"], state["v"], state["m"], case["steps"], state["G"], state["dt"],
                                     case["precision"], case["ckpt"])
        loss = (rt[:, state["idx"]] - state["target"]).square().sum()
        g = torch.autograd.grad(loss, (state["r"], state["v"], state["m"]))
        return {"r": rt.detach(), "v": vt.detach().to(kept), "dr0": g[0].to(kept), "dv0": g[1].to(kept),
                "dm": g[2].to(kept)}
    sim = state["sim"]
    if kind == "energy":
        return sim.energy()
    if kind == "grad":
        return dict(zip(("dr0", "dv0", "dm"), (g.to(kept) for g in sim.grad(case["steps"], state["dr"]))))
    sim.step(case["steps"])
    return {"r": sim.r, "v": sim.v.to(kept), "a": sim.accel().to(kept)}


def work(case):
    """Each unordered pair once -- 3 differences, 5 for |d|^2, 3 for |d|^-3, 2 mass products and 12 for the two
    accumulated terms -- and each array of the state read or written once."""
    if "systems" in case:
        mean = 0.5 * (case["lo"] + case["hi"])
        bodies, pairs = case["systems"] * mean, case["systems"] * mean * mean / 2
    else:
        bodies, pairs = case["n"], case["n"] * (case["n"] - 1) / 2
    kind, steps = case["kind"], case.get("steps", 1)
    if kind == "energy":  # 3 + 5 + 1, the two masses, the sum
        return {"bytes": 56.0 * bodies, "flops": 12.0 * pairs}
    if kind == "static":
        return {"bytes": 56.0 * bodies, "flops": 25.0 * pairs}
    if kind == "step":
        evals = steps * (4 if case.get("integrator") == "rk4" else 1)
        return {"bytes": 128.0 * bodies, "flops": 25.0 * pairs * evals}
    # forward (also run by grad), and one vector-Jacobian product per step and one at r0 (58 per pair)
    return {"bytes": 136.0 * bodies, "flops": 25.0 * pairs * steps + 58.0 * pairs * (steps + 1)}


# ---------------------------------------------------------------------------
# The same results in plain torch, FP64
# ---------------------------------------------------------------------------
def _tensors(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    systems = _systems(case, seed)
    off, r, v, m = inputs.concat(systems)
    return systems[0], off, *(torch.tensor(t, device=dev) for t in (r, v, m))


def _chunks(n):
    step = max(1, (1 << 25) // n)
    return [(b, min(n, b + step)) for b in range(0, n, step)]


def _pairs(r, b, e):
    """Differences r_j - r_p of targets [b, e) and |d|^-1 (0 for the target itself)."""
    d = r[:, None, :] - r[:, b:e, None]
    r2 = (d * d).sum(0)
    k = torch.arange(b, e, device=r.device)
    r2[k - b, k] = math.inf
    return d, 1.0 / r2.sqrt()


def _accel(r, mu):
    a = torch.empty_like(r)
    for b, e in _chunks(r.shape[1]):
        d, y = _pairs(r, b, e)
        a[:, b:e] = (d * (mu * y * y * y)).sum(2)
    return a


def _accel_of(off, mu):
    def f(r):
        return torch.cat([_accel(r[:, b:e], mu[b:e]) for b, e in zip(off[:-1], off[1:])], 1)
    return f


def _vjp(r, mu, w):
    """(J^T w [3, n], sum_j |d|^-3 (w_j . d) [n]) of Eq. 1 at r."""
    jt, gs = torch.empty_like(r), torch.empty_like(r[0])
    for b, e in _chunks(2 * r.shape[1]):
        e = min(e, r.shape[1])
        if b >= e:
            break
        d, y = _pairs(r, b, e)
        y3 = y * y * y
        u = mu[None, b:e, None] * w[:, None, :] - mu * w[:, b:e, None]
        jt[:, b:e] = (y3 * u - 3.0 * (y3 * y * y * (d * u).sum(0)) * d).sum(2)
        gs[b:e] = (y3 * (w[:, None, :] * d).sum(0)).sum(1)
    return jt, gs


def _verlet(f, r, v, dt, steps, path=None):
    a = f(r)
    for _ in range(steps):
        if path is not None:
            path.append(r)
        r = r + v * dt + (0.5 * dt * dt) * a
        an = f(r)
        v = v + (0.5 * dt) * (a + an)
        a = an
    if path is not None:
        path.append(r)
    return r, v, a


def _gradient(path, mu, G, dt, steps, rho, nu):
    """Reverse sweep of the discrete Verlet recurrence from (rho, nu) = dL/d(r_T, v_T)."""
    gm = torch.zeros_like(mu)
    w = (0.5 * dt) * nu
    for i in range(steps - 1, -1, -1):
        jt, gs = _vjp(path[i + 1], mu, w)
        rho, gm = rho + jt, gm - G * gs
        nun = nu + dt * rho
        w = (0.5 * dt * dt) * rho + (0.5 * dt) * nu + ((0.5 * dt) * nun if i > 0 else 0.0)
        nu = nun
    jt, gs = _vjp(path[0], mu, w)
    return rho + jt, nu, gm - G * gs


def _close_steps(s, r, v, m, mu, steps):
    """Close pairs (omega dt > theta_c at the start) sub-cycled, everything else by Verlet with the far force."""
    dt, n = s.dt, s.n
    pairs = []
    for b, e in _chunks(n):
        y = _pairs(r, b, e)[1]
        hit = (mu[None, :] + mu[b:e, None]) * dt * dt * y**3 > CLOSE[0] ** 2
        p, j = (t.cpu().numpy() for t in hit.nonzero(as_tuple=True))
        pairs += [(int(x) + b, int(z)) for x, z in zip(p, j) if x + b < z]
    root = list(range(n))

    def find(x):
        while root[x] != x:
            x = root[x]
        return x

    for p, j in pairs:
        root[find(p)] = find(j)
    clusters = {}
    for p, j in pairs:
        clusters.setdefault(find(p), []).append((p, j))
    pp = torch.tensor(pairs, dtype=torch.long, device=r.device).reshape(-1, 2).T
    rn, mn = r.cpu().numpy(), mu.cpu().numpy()
    plan = []
    for pr in clusters.values():
        mem = sorted({x for q in pr for x in q})
        at = {x: i for i, x in enumerate(mem)}
        om = max(math.sqrt((mn[p] + mn[j]) / np.linalg.norm(rn[:, j] - rn[:, p]) ** 3) * dt for p, j in pr)
        plan.append((np.array(mem), np.array([[at[p], at[j]] for p, j in pr]).T, math.ceil(om / CLOSE[1])))

    def near(x, mk, ab):
        d = x[:, ab[1]] - x[:, ab[0]]
        s3 = (d * d).sum(0) ** -1.5
        out = np.zeros_like(x)
        np.add.at(out, (slice(None), ab[0]), d * (mk[ab[1]] * s3))
        np.add.at(out, (slice(None), ab[1]), -d * (mk[ab[0]] * s3))
        return out

    def far(x):  # members: every body but themselves and their close partners
        a = _accel(x, mu)
        for mem, ab, _ in plan:
            for i, p in enumerate(mem):
                d = x - x[:, p : p + 1]
                y = 1.0 / (d * d).sum(0).sqrt()
                out = [p] + [mem[k] for k in np.concatenate([ab[1][ab[0] == i], ab[0][ab[1] == i]])]
                y[torch.tensor([int(k) for k in out], device=y.device)] = 0.0
                a[:, p] = (d * (mu * y * y * y)).sum(1)
        return a

    af = far(r)
    for _ in range(steps):
        vh = v + (0.5 * dt) * af
        rnew, vnew = r + dt * vh, vh.clone()
        for mem, ab, k in plan:
            q = torch.tensor(mem, device=r.device)
            x, u, mk, h = r[:, q].cpu().numpy(), vh[:, q].cpu().numpy(), mn[mem], dt / k
            a = near(x, mk, ab)
            for _ in range(k):
                u = u + (0.5 * h) * a
                x = x + h * u
                a = near(x, mk, ab)
                u = u + (0.5 * h) * a
            rnew[:, q], vnew[:, q] = torch.tensor(x, device=r.device), torch.tensor(u, device=r.device)
        r = rnew
        af = far(r)
        v = vnew + (0.5 * dt) * af
    return r, v


def exact(case, seed):
    kind, steps = case["kind"], case.get("steps", 1)
    if case.get("n", 0) > 70000:
        return None  # the plain evaluation of N^2 pairs takes too long
    s, off, r, v, m = _tensors(case, seed)
    dt, mu = s.dt, s.G * m
    if kind == "static":
        return _accel(r, mu)
    if kind == "energy":
        pot = torch.zeros((), dtype=r.dtype, device=r.device)
        for b, e in _chunks(s.n):
            pot = pot - 0.5 * (m[b:e] * (mu * _pairs(r, b, e)[1]).sum(1)).sum()
        return np.array([float(0.5 * (m * (v * v).sum(0)).sum() + pot)])
    if case.get("close"):
        r, v = _close_steps(s, r, v, m, mu, steps)
        return {"r": r, "v": v, "a": _accel(r, mu)}
    f = _accel_of(off, mu)
    if kind in ("grad", "train"):
        idx, target = _loss(case, seed, s)
        target = torch.tensor(target, device=r.device)
        path = []
        rt, vt, _ = _verlet(f, r, v, dt, steps, path)
        rho = torch.zeros_like(r)
        rho[:, idx] = 2.0 * ((rt if kind == "train" else r)[:, idx] - target)
        g = dict(zip(("dr0", "dv0", "dm"), _gradient(path, mu, s.G, dt, steps, rho, torch.zeros_like(r))))
        return dict(g, r=rt, v=vt) if kind == "train" else g
    integrator = case.get("integrator", "verlet")
    if integrator == "verlet":
        r, v, a = _verlet(f, r, v, dt, steps)
    elif integrator == "leapfrog":
        for _ in range(steps):
            h = r + (0.5 * dt) * v
            a = f(h)  # the acceleration that the integrator keeps: at the half step
            v = v + dt * a
            r = h + (0.5 * dt) * v
    else:
        for _ in range(steps):
            k1, l1 = v, f(r)
            k2, l2 = v + (0.5 * dt) * l1, f(r + (0.5 * dt) * k1)
            k3, l3 = v + (0.5 * dt) * l2, f(r + (0.5 * dt) * k2)
            k4, l4 = v + dt * l3, f(r + dt * k3)
            r = r + (dt / 6.0) * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
            v = v + (dt / 6.0) * (l1 + 2.0 * l2 + 2.0 * l3 + l4)
        a = f(r)
    return {"r": r, "v": v, "a": a}
