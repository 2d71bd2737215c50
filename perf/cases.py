"""The work that a program using this library has it do, as cases that can be timed.

Every case goes through the package's public entry points: leapfrog steps of
one system (nbody_step) and of a forest (nbody_step_batched), single force
evaluations (nbody_build + nbody_walk), the direct sum (nbody_direct) and the
cost model's forward and backward pass (nbody_mlp_eval).  Inputs are sampled on
the GPU from the seed: Plummer and Hernquist spheres and the bulge + disk +
halo galaxy of the benchmark (G = 1, total mass 1, equal masses, dt = 1/256).
"""
import math

import numpy as np
import torch

import paper_1811_02761_gb300 as nb

_TWO_PI = 2.0 * math.pi


def listed():
    return [
        # a small cluster followed for many steps from a captured step graph:
        # launch latency and short kernels decide
        {"name": "step-plummer-4k", "kind": "step", "model": "plummer", "n": 4096, "steps": 16,
         "graph": 1, "rebuild": 1, "levels": 0, "host": 0},
        # an ordinary run with the default parameters (eager steps), odd count
        {"name": "step-galaxy-100k", "kind": "step", "model": "galaxy", "n": 100003, "steps": 4,
         "graph": 0, "rebuild": 1, "levels": 0, "host": 0},
        # a program that keeps its state in page-locked host memory and takes
        # one step per call (the benchmark's end-to-end measurement)
        {"name": "step-galaxy-1m-host", "kind": "step", "model": "galaxy", "n": 1000003, "steps": 1,
         "graph": 0, "rebuild": 1, "levels": 0, "host": 1},
        # the headline workload: the largest galaxy, step graph
        {"name": "step-galaxy-8m", "kind": "step", "model": "galaxy", "n": 1 << 23, "steps": 5,
         "graph": 1, "rebuild": 1, "levels": 0, "host": 0},
        # block time steps with the tree refitted between rebuilds, as the
        # paper's code runs; dt = 1/8
        {"name": "step-hernquist-block", "kind": "step", "model": "hernquist", "n": 65539, "steps": 1,
         "graph": 0, "rebuild": 4, "levels": 6, "host": 0},
        # the many-system workload: 512 systems of 2^10 .. 2^16 particles
        {"name": "forest-512", "kind": "forest", "systems": 512, "log2_min": 10.0, "log2_max": 16.0,
         "steps": 3, "graph": 1, "schedule": 0},
        # fewer and smaller systems, walk queue ordered by the learned cost model
        {"name": "forest-96-learned", "kind": "forest", "systems": 96, "log2_min": 10.0,
         "log2_max": 14.0, "steps": 2, "graph": 0, "schedule": 1},
        # forces and potential of a snapshot, nothing known about |a| yet
        {"name": "force-plummer-first", "kind": "force", "model": "plummer", "n": 262147,
         "log2_dacc": -9, "quad": 0, "phi": 1, "first": 1},
        # forces with quadrupole moments, |a| known from the step before
        {"name": "force-galaxy-quad", "kind": "force", "model": "galaxy", "n": 300007,
         "log2_dacc": -12, "quad": 1, "phi": 0, "first": 0},
        # a precise force evaluation (compensated sums), small odd system
        {"name": "force-hernquist-tight", "kind": "force", "model": "hernquist", "n": 30011,
         "log2_dacc": -20, "quad": 0, "phi": 1, "first": 0},
        # the direct sum a program checks its tree forces against
        {"name": "direct-plummer-50k", "kind": "direct", "model": "plummer", "n": 50021,
         "compensated": 1, "phi": 1},
        # prediction, loss and gradient of the cost model over one walk's groups
        {"name": "cost-model-60k", "kind": "model", "n": 60013},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "forest", "force", "force", "direct", "model"])
    model = rng.choice(["plummer", "hernquist", "galaxy"])
    if kind == "step":
        levels = rng.choice([0, 0, 0, 6])
        host = 0 if levels else rng.choice([0, 0, 1])
        return {"kind": kind, "model": model,
                "n": _log_int(rng, 1000, 100000 if levels else 4000000),
                "steps": 1 if levels or host else rng.randint(2, 8),
                "graph": 0 if levels or host else rng.choice([0, 1]),
                "rebuild": rng.choice([1, 1, 4]), "levels": levels, "host": host}
    if kind == "forest":
        lo = rng.uniform(9.0, 11.0)
        return {"kind": kind, "systems": _log_int(rng, 16, 400), "log2_min": lo,
                "log2_max": lo + rng.uniform(1.0, 4.0), "steps": rng.randint(1, 3),
                "graph": rng.choice([0, 1]), "schedule": rng.choice([0, 0, 1])}
    if kind == "force":
        dacc = rng.choice([-7, -9, -9, -12, -20])
        return {"kind": kind, "model": model,
                "n": _log_int(rng, 1000, 60000 if dacc == -20 else 1000000), "log2_dacc": dacc,
                "quad": rng.choice([0, 0, 1]), "phi": rng.choice([0, 1]),
                "first": rng.choice([0, 1])}
    if kind == "direct":
        return {"kind": kind, "model": model, "n": _log_int(rng, 500, 100000),
                "compensated": rng.choice([0, 1]), "phi": rng.choice([0, 1])}
    return {"kind": kind, "n": _log_int(rng, 1000, 250000)}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _normal(g, n):
    return torch.randn(n, generator=g, device="cuda", dtype=torch.float64)


def _isotropic(g, r):
    n = r.numel()
    c = _uniform(g, n, -1.0, 1.0)
    s = torch.sqrt((1.0 - c * c).clamp_min(0.0))
    p = _uniform(g, n, 0.0, _TWO_PI)
    return torch.stack([r * s * torch.cos(p), r * s * torch.sin(p), r * c])


def _plummer(g, n):
    """Scale radius 1, cut at 64; Gaussian velocities of the local dispersion."""
    cut = (1.0 + 64.0 ** -2) ** -1.5
    r = (_uniform(g, n, 1e-9, cut) ** (-2.0 / 3.0) - 1.0).clamp_min(1e-12) ** -0.5
    v = torch.stack([_normal(g, n) for _ in range(3)]) * torch.sqrt(1.0 / (6.0 * torch.sqrt(1.0 + r * r)))
    return _isotropic(g, r), v


def _hernquist(g, n, a=1.0):
    """Cut at 100 a; Gaussian velocities of about the Jeans dispersion."""
    s = torch.sqrt(_uniform(g, n, 0.0, (100.0 / 101.0) ** 2))
    r = a * s / (1.0 - s)
    v = torch.stack([_normal(g, n) for _ in range(3)]) * torch.sqrt(r / (r + a) ** 2 / 4.0)
    return _isotropic(g, r), v


def _inverse(f, lo, hi, u, points=8192):
    """x with f(x) = u f(hi) for the increasing f with f(lo) = 0, from a table."""
    t = torch.linspace(0.0, 1.0, points, device="cuda", dtype=torch.float64)
    x = lo + (hi - lo) * t * t
    y = f(x) / f(x)[-1]
    k = torch.searchsorted(y, u).clamp(1, points - 1)
    w = ((u - y[k - 1]) / (y[k] - y[k - 1])).clamp(0.0, 1.0)
    return x[k - 1] + w * (x[k] - x[k - 1])


def _galaxy(g, n):
    """Hernquist bulge (15 %, a = 0.6), exponential disk (10 %, R_d = 5.4),
    NFW halo (75 %, r_s = 12, cut at 10 r_s), shuffled together."""
    nbulge, ndisk = round(0.15 * n), round(0.10 * n)
    nhalo = n - nbulge - ndisk
    nfw = lambda t: torch.log1p(t) - t / (1.0 + t)  # noqa: E731
    disk = lambda t: 1.0 - (1.0 + t) * torch.exp(-t)  # noqa: E731

    def mass(r):
        return (0.15 * (r / (r + 0.6)) ** 2 + 0.10 * disk((r / 5.4).clamp_max(10.0)) +
                0.75 * nfw((r / 12.0).clamp_max(10.0)) / nfw(torch.full_like(r, 10.0)))

    xb, vb = _hernquist(g, nbulge, 0.6)
    rh = 12.0 * _inverse(nfw, 0.0, 10.0, _uniform(g, nhalo))
    xh = _isotropic(g, rh)
    vh = torch.stack([_normal(g, nhalo) for _ in range(3)]) * torch.sqrt(mass(rh) / (3.0 * rh.clamp_min(1e-3)))
    R = 5.4 * _inverse(disk, 0.0, 10.0, _uniform(g, ndisk))
    z = 0.6 * torch.atanh(_uniform(g, ndisk, -1.0 + 1e-4, 1.0 - 1e-4))
    p = _uniform(g, ndisk, 0.0, _TWO_PI)
    vc = torch.sqrt(mass(R) / R.clamp_min(1e-3))
    vr, vp = 0.1 * vc * _normal(g, ndisk), vc * (1.0 + 0.1 * _normal(g, ndisk))
    xd = torch.stack([R * torch.cos(p), R * torch.sin(p), z])
    vd = torch.stack([vr * torch.cos(p) - vp * torch.sin(p), vr * torch.sin(p) + vp * torch.cos(p),
                      0.05 * vc * _normal(g, ndisk)])
    k = torch.randperm(n, generator=g, device="cuda")
    return torch.cat([xb, xd, xh], 1)[:, k], torch.cat([vb, vd, vh], 1)[:, k]


def _sample(model, n, seed):
    """Positions (FP64), velocities, masses and softening of one system."""
    x, v = {"plummer": _plummer, "hernquist": _hernquist, "galaxy": _galaxy}[model](_gen(seed), n)
    m = torch.full((n,), 1.0 / n, device="cuda", dtype=torch.float32)
    return x, v.float(), m, 1.0 / 64 if model == "galaxy" else 1.0 / 128


def _forest(case, seed):
    """Systems of log-uniform size (the case's own, so that every seed has the
    same count), Plummer or Hernquist, eps = 4 / N^(1/3)."""
    r = np.random.default_rng(case["systems"])
    sizes = np.rint(2.0 ** r.uniform(case["log2_min"], case["log2_max"], case["systems"])).astype(np.int64)
    r = np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    g = _gen(seed)
    plummer = torch.from_numpy(np.repeat(r.integers(0, 2, sizes.size), sizes).astype(bool)).cuda()
    xp, vp = _plummer(g, n)
    xh, vh = _hernquist(g, n)
    m = torch.from_numpy(np.repeat(1.0 / sizes, sizes).astype(np.float32)).cuda()
    eps = (4.0 / sizes ** (1.0 / 3.0)).astype(np.float32)
    return torch.where(plummer, xp, xh), torch.where(plummer, vp, vh).float(), m, off, eps


class _Context:
    """A library context that is given back with the state that holds it."""

    def __init__(self, **config):
        self.handle = nb.nbody_create(nb.nbody_config_default(**config))

    def __del__(self):
        nb.nbody_destroy(self.handle)


def _rows(t):
    return [t[k].contiguous() for k in range(t.shape[0])]


def _empty(n, count=3):
    return [torch.empty(n, device="cuda", dtype=torch.float32) for _ in range(count)]


def _dt(case):
    return 1.0 / 8 if case.get("levels") else 1.0 / 256


def prepare(case, seed):
    kind = case["kind"]
    if kind == "model":
        g = _gen(seed)
        n = case["n"]
        f = (_normal(g, 8 * n).reshape(n, 8) * 2.0 + 1.0).float().contiguous()
        t = (f.double() @ _uniform(g, 8, -0.3, 0.3) + 0.1 * _normal(g, n)).float()
        w = (_uniform(g, nb.MLP_PARAMS, -1.0, 1.0) * 0.3).float()
        norm = torch.cat([torch.full((8,), 1.0), torch.full((8,), 2.0)]).cuda()
        return {"kind": kind, "features": f, "targets": t, "params": w, "norm": norm}
    if kind == "forest":
        x, v, m, off, eps = _forest(case, seed)
        n = m.numel()
        ctx = _Context(use_graph=case["graph"])
        a = _empty(n)
        nb.nbody_build_batched(ctx.handle, off, eps, *_rows(x.float()), m)
        nb.nbody_walk(ctx.handle, None, *a)
        if case["schedule"] == nb.SCHED_MLP:  # trained on the costs of the first walk
            g = _gen(seed + 1)
            nb.nbody_mlp_set_params(ctx.handle, (_uniform(g, nb.MLP_PARAMS, -1.0, 1.0) * 0.4).float())
            nb.nbody_mlp_train(ctx.handle, 20, 1e-2, 4096)
            cfg = nb.nbody_get_config(ctx.handle)
            cfg.schedule = nb.SCHED_MLP
            nb.nbody_set_config(ctx.handle, cfg)
        return {"kind": kind, "ctx": ctx, "off": off, "eps": eps, "x": _rows(x), "v": _rows(v),
                "m": m, "a": a, "dt": _dt(case), "steps": case["steps"]}
    x, v, m, eps = _sample(case["model"], case["n"], seed)
    n = case["n"]
    if kind == "direct":
        return {"kind": kind, "x": _rows(x.float()), "m": m, "eps": eps,
                "compensated": case["compensated"], "out": _empty(n, 4 if case["phi"] else 3)}
    if kind == "force":
        ctx = _Context(eps=eps, delta_acc=2.0 ** case["log2_dacc"], quadrupole=case["quad"],
                       want_potential=case["phi"])
        xf, aold = _rows(x.float()), None
        if not case["first"]:  # |a| of the step before: a walk with the default parameters
            a, c = _empty(n), _Context(eps=eps)
            nb.nbody_build(c.handle, *xf, m)
            nb.nbody_walk(c.handle, None, *a)
            aold = torch.sqrt(a[0] ** 2 + a[1] ** 2 + a[2] ** 2)
        return {"kind": kind, "ctx": ctx, "x": xf, "m": m, "aold": aold,
                "out": _empty(n, 4 if case["phi"] else 3)}
    ctx = _Context(eps=eps, use_graph=case["graph"], rebuild_interval=case["rebuild"],
                   block_levels=case["levels"])
    a = _empty(n)
    nb.nbody_build(ctx.handle, *_rows(x.float()), m)
    nb.nbody_walk(ctx.handle, None, *a)
    s = {"kind": kind, "ctx": ctx, "x": _rows(x), "v": _rows(v), "m": m, "a": a, "dt": _dt(case),
         "steps": case["steps"]}
    if case["host"]:
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)  # noqa: E731
        s.update(x=[pin(t) for t in s["x"]], v=[pin(t) for t in s["v"]], a=[pin(t) for t in a],
                 m=pin(m))
    return s


# ---------------------------------------------------------------- one pass
def run(state):
    s = state
    if s["kind"] == "step":
        nb.nbody_step(s["ctx"].handle, *s["x"], *s["v"], s["m"], *s["a"], s["dt"], s["steps"])
        return {"x": s["x"], "v": s["v"], "a": s["a"]}
    if s["kind"] == "forest":
        nb.nbody_step_batched(s["ctx"].handle, s["off"], s["eps"], *s["x"], *s["v"], s["m"], *s["a"],
                              s["dt"], s["steps"])
        return {"x": s["x"], "v": s["v"], "a": s["a"]}
    if s["kind"] == "force":
        nb.nbody_build(s["ctx"].handle, *s["x"], s["m"])
        nb.nbody_walk(s["ctx"].handle, s["aold"], *s["out"])
        return {"out": s["out"]}
    if s["kind"] == "direct":
        nb.nbody_direct(*s["x"], s["m"], 1.0, s["eps"], s["compensated"], *s["out"])
        return {"out": s["out"]}
    pred, grad, loss = nb.nbody_mlp_eval(s["features"], s["targets"], s["params"], s["norm"])
    return {"pred": pred, "grad": grad, "loss": loss}


# ---------------------------------------------------------------- what a pass cannot do without
def _interactions(n, log2_dacc):
    """List entries per particle, about: 1500 at delta_acc = 2^-9, and 40 times
    as many at 2^-20 (measured on the galaxy), never more than the particles."""
    return min(n, 1500.0 * 2.0 ** (0.485 * (-9 - log2_dacc)))


def work(case):
    kind = case["kind"]
    if kind == "model":  # 8 -> 32 -> 32 -> 1, forward and both backward products
        return {"bytes": case["n"] * 40.0 + 3 * 4 * nb.MLP_PARAMS, "flops": case["n"] * 6.0 * 1312}
    if kind == "direct":
        return {"bytes": case["n"] * (16.0 + 12.0 + 4.0 * case["phi"]), "flops": 22.0 * case["n"] ** 2}
    if kind == "force":
        inter = case["n"] * _interactions(case["n"], case["log2_dacc"])
        return {"bytes": case["n"] * (28.0 + 4.0 * case["phi"] + (0.0 if case["first"] else 4.0)),
                "flops": 22.0 * inter * (2.0 if case["first"] else 1.0)}
    if kind == "forest":
        lo, hi = case["log2_min"], case["log2_max"]
        n = case["systems"] * (2.0 ** hi - 2.0 ** lo) / ((hi - lo) * math.log(2.0))
        inter = n * _interactions(2.0 ** (0.5 * (lo + hi)), -9)
    else:
        n = float(case["n"])
        inter = n * _interactions(n, -9)
    # position (FP64), velocity, mass, acceleration in; position, velocity, acceleration out
    return {"bytes": n * (52.0 + 48.0), "flops": 22.0 * inter * case["steps"]}


# ---------------------------------------------------------------- the same in 64 bits
_MOST_PAIRS = 1.0e11


def _direct64(x, m, eps):
    """Eq. 1 and the potential of every particle by direct summation in FP64."""
    n = m.numel()
    a, phi = torch.empty_like(x), torch.empty_like(m)
    rows = max(1, min(n, (1 << 27) // n))
    for lo in range(0, n, rows):
        hi = min(n, lo + rows)
        d = [x[k][None, :] - x[k][lo:hi, None] for k in range(3)]
        w = torch.rsqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps)
        phi[lo:hi] = -(w @ m) + m[lo:hi] / eps
        w = w * w * w
        for k in range(3):
            a[k, lo:hi] = (w * d[k]) @ m
    return a, phi


def _exact_model(case, seed):
    s = prepare(case, seed)
    w = s["params"].to(torch.bfloat16).double()
    w1, b1, w2, b2, w3, b3 = (t.clone().requires_grad_() for t in (
        w[:256].reshape(8, 32), w[256:288], w[288:1312].reshape(32, 32), w[1312:1344], w[1344:1376],
        w[1376:]))
    x = (s["features"].double() - s["norm"][:8].double()) / s["norm"][8:].double()
    pred = torch.relu(torch.relu(x @ w1 + b1) @ w2 + b2) @ w3 + b3
    loss = ((pred - s["targets"].double()) ** 2).mean()
    grads = torch.autograd.grad(loss, (w1, b1, w2, b2, w3, b3))
    return {"pred": pred.detach(), "grad": torch.cat([g.reshape(-1) for g in grads]),
            "loss": float(loss)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "model":
        return _exact_model(case, seed)
    if kind == "forest":
        return None
    x, v, m, eps = _sample(case["model"], case["n"], seed)
    n, m = case["n"], m.double()
    eps = float(np.float32(eps))
    if kind in ("direct", "force"):
        if float(n) * n > _MOST_PAIRS:
            return None
        a, phi = _direct64(x.float().double(), m, eps)
        return {"out": [a[0], a[1], a[2]] + ([phi] if case["phi"] else [])}
    if case["levels"] or float(n) * n * (case["steps"] + 1) > _MOST_PAIRS:
        return None
    x, v, dt = x.clone(), v.double(), _dt(case)
    a, _ = _direct64(x, m, eps)
    for _ in range(case["steps"]):  # kick, drift, kick
        v = v + 0.5 * dt * a
        x = x + dt * v
        a, _ = _direct64(x, m, eps)
        v = v + 0.5 * dt * a
    return {"x": list(x), "v": list(v), "a": list(a)}
