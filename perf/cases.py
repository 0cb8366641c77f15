"""Performance cases: what a user of this package has it do, through its public calls.

``listed()`` holds the fixed cases, ``draw(rng)`` one more of the same ranges,
``prepare(case, seed)`` the inputs and the context (autotuned, as ``nbody_init``
leaves it), ``run(state)`` one pass, ``work(case)`` the bytes and operations a
pass needs and ``exact(case, seed)`` the same results from plain float64 torch.

Kinds of cases:

* ``forces``   -- ``nbody_forces`` with potentials, one system;
* ``step``     -- ``nbody_step`` continuing a trajectory (a valid on entry);
* ``host``     -- ``nbody_step_host`` on pinned host arrays;
* ``ensemble`` -- ``nbody_step`` of many systems in one context, replayed as a CUDA graph;
* ``noalloc``  -- ``nbody_forces_noalloc``;
* ``train``    -- forward and backward through ``NBodyAdjoint``;
* ``adjoint``  -- ``nbody_adjoint_params`` with given final gradients.

Bodies are Plummer spheres of equal masses, pairs of spheres with log-normal
masses, or the Lennard-Jones gas, from ``inputs``. The mixed path's arithmetic
is float32, so its results are handed on as float32, the way snapshots are
written and optimisers take gradients; FP64 results are returned as they are.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2511_02655_gb300 as nb
from paper_2511_02655_gb300 import inputs

DEV = "cuda:0"


def _case(name, kind, n, **kw):
    c = dict(name=name, kind=kind, n=n, precision="mixed", law="gravity", masses="equal", eps=0.01, dt=1e-3,
             steps=1, every=0, graph=False, checkpoint=0, systems=1, layout=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call in earnest: one force evaluation of a small sphere, latency and launches
        _case("forces_mixed_1024", "forces", 1024),
        # one force evaluation of a medium system with unequal masses at a size no tile divides
        _case("forces_mixed_10007", "forces", 10007, masses="lognormal", eps=0.02),
        # a large collision model, two spheres with log-normal masses: pair throughput
        _case("forces_mixed_262144", "forces", 262144, masses="lognormal", eps=0.002),
        # the headline workload: one step with its energy record
        _case("step_mixed_65536", "step", 65536, eps=0.005, dt=5e-4, every=1),
        # many uneven systems in one context, replayed as a graph, energies at the end
        _case("ensemble_mixed_128", "ensemble", 16384, steps=10, every=10, graph=True, systems=128, layout=4),
        # the paper's Lennard-Jones gas between walls, energy every step
        _case("lj_mixed_10000", "step", 10000, law="lj", eps=0.0, dt=5e-3, steps=20, every=1, graph=True),
        # a simulation whose state lives in host memory: copies both ways and one step
        _case("host_mixed_32768", "host", 32768, eps=0.005, dt=5e-4, every=1),
        # forces where nothing may be allocated, ragged size
        _case("noalloc_mixed_20001", "noalloc", 20001, masses="lognormal", eps=0.02),
        # gradients of a final-state loss, forward and backward
        _case("train_mixed_16384", "train", 16384, steps=40, checkpoint=20),
        # the plain method: ten steps in FP64 with energies
        _case("step_fp64_1024", "step", 1024, precision="fp64", steps=10, every=1),
        # an FP64 force evaluation of a medium system, unequal masses, ragged
        _case("forces_fp64_12002", "forces", 12002, precision="fp64", masses="lognormal", eps=0.02),
        # FP64 gradients with those of G and eps
        _case("adjoint_fp64_2048", "adjoint", 2048, precision="fp64", masses="lognormal", eps=0.05, steps=20,
              checkpoint=10),
    ]


def _log_size(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["forces", "forces", "step", "step", "lj", "ensemble", "host", "noalloc", "train", "forces64",
                       "step64", "lj64", "adjoint64"])
    masses = rng.choice(["equal", "lognormal"])
    eps = rng.choice([0.005, 0.01, 0.02, 0.05])
    if kind == "forces":
        c = _case("", "forces", _log_size(rng, 64, 200000), masses=masses, eps=eps)
    elif kind == "step":
        c = _case("", "step", _log_size(rng, 64, 100000), masses=masses, eps=eps, steps=rng.choice([1, 2, 5]),
                  every=rng.choice([0, 1]), graph=rng.choice([False, True]))
    elif kind == "lj":
        c = _case("", "step", _log_size(rng, 500, 30000), law="lj", eps=0.0, dt=5e-3, steps=rng.choice([5, 20]),
                  every=rng.choice([0, 1]), graph=rng.choice([False, True]))
    elif kind == "ensemble":
        c = _case("", "ensemble", rng.choice([2048, 8192, 16384]), masses="equal", eps=eps, steps=5, every=5,
                  graph=rng.choice([False, True]), systems=rng.randint(8, 128), layout=rng.randint(0, 1 << 20))
    elif kind == "host":
        c = _case("", "host", _log_size(rng, 256, 65536), masses=masses, eps=eps, dt=5e-4, every=1,
                  graph=rng.choice([False, True]))
    elif kind == "noalloc":
        c = _case("", "noalloc", _log_size(rng, 64, 100000), masses=masses, eps=eps)
    elif kind == "train":
        c = _case("", "train", _log_size(rng, 256, 16384), masses=masses, eps=eps, steps=rng.choice([10, 30]),
                  checkpoint=rng.choice([5, 10]))
    elif kind == "forces64":
        c = _case("", "forces", _log_size(rng, 64, 12000), precision="fp64", masses=masses, eps=eps)
    elif kind == "step64":
        c = _case("", "step", _log_size(rng, 64, 8192), precision="fp64", masses=masses, eps=eps,
                  steps=rng.choice([1, 4]), every=1)
    elif kind == "lj64":
        c = _case("", "step", _log_size(rng, 500, 10000), precision="fp64", law="lj", eps=0.0, dt=5e-3, steps=2,
                  every=1)
    else:
        c = _case("", "adjoint", _log_size(rng, 128, 3000), precision="fp64", masses=masses, eps=0.05,
                  steps=rng.choice([5, 10]), checkpoint=5)
    if c["masses"] == "lognormal":
        c["n"] += c["n"] % 2 if c["kind"] != "noalloc" else 0
    del c["name"]
    return c


def _bodies(case, seed):
    """(x, v, m, box, offsets) as float64 host arrays."""
    n = case["n"]
    if case["kind"] == "ensemble":
        sizes = inputs.ensemble_sizes(case["systems"], case["layout"], 64, n)
        ens = inputs.ensemble(len(sizes), seed, sizes=sizes)
        return ens.x, ens.v, ens.m, 0.0, [int(o) for o in ens.offsets]
    if case["law"] == "lj":
        x, v, m, box = inputs.lj_gas(n, seed)
        return x, v, m, box, [0, n]
    if case["masses"] == "lognormal":
        x, v, m = inputs.two_spheres(n + n % 2, seed)
        x, v, m = x[:n], v[:n], m[:n]
    else:
        x, v, m = inputs.plummer(n, seed)
    return x, v, m, 0.0, [0, n]


def _context(case, box, offsets):
    return nb.nbody_init(G=1.0, eps=case["eps"], dt=case["dt"], offsets=offsets, energy_every=case["every"],
                         precision=nb.FP64 if case["precision"] == "fp64" else nb.MIXED,
                         law=nb.LENNARD_JONES if case["law"] == "lj" else nb.GRAVITY, box=box,
                         flags=nb.FLAG_GRAPH if case["graph"] else 0)


class _Arrays:
    """Named float64 arrays in one block, so that one conversion hands all of them on."""

    def __init__(self, shapes, device, mixed, pinned=False):
        self.mixed, self.at, total = mixed, {}, 0
        for name, shape in shapes.items():
            self.at[name] = (total, shape)
            total += math.prod(shape)
        self.block = torch.zeros(total, dtype=torch.float64, device=device, pin_memory=pinned)

    def _view(self, block, name):
        lo, shape = self.at[name]
        return block[lo:lo + math.prod(shape)].view(shape)

    def __getitem__(self, name):
        return self._view(self.block, name)

    def handed_on(self):
        block = self.block.float() if self.mixed else self.block
        return {name: self._view(block, name) for name in self.at}


def prepare(case, seed):
    x, v, m, box, offsets = _bodies(case, seed)
    n, kind, mixed = offsets[-1], case["kind"], case["precision"] == "mixed"
    s = {"case": case, "n": n, "m": torch.from_numpy(np.ascontiguousarray(m)).to(DEV)}
    if kind != "noalloc":
        s["ctx"] = _context(case, box, offsets)
    if kind in ("forces", "noalloc"):
        s["x"] = torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
        s["out"] = _Arrays({"a": (n, 3), "phi": (n,)}, DEV, mixed)
    elif kind in ("step", "ensemble", "host"):
        shapes = {"x": (n, 3), "v": (n, 3), "a": (n, 3)}
        if case["every"]:
            shapes["log"] = (case["steps"] // case["every"], len(offsets) - 1, 9)
        s["out"] = _Arrays(shapes, "cpu" if kind == "host" else DEV, mixed, pinned=kind == "host")
        s["out"]["x"].copy_(torch.from_numpy(x))
        s["out"]["v"].copy_(torch.from_numpy(v))
        a, _ = nb.nbody_forces(s["ctx"], torch.from_numpy(x).to(DEV), s["m"], with_phi=False)
        s["out"]["a"].copy_(a)
        if kind == "host":
            s["m"] = s["m"].cpu().pin_memory()
    else:
        rng = np.random.default_rng(seed + 1)
        s["x"], s["v"] = (torch.from_numpy(np.ascontiguousarray(t)).to(DEV) for t in (x, v))
        if kind == "train":
            s["target"] = torch.from_numpy(inputs.targets(n, seed + 1)).to(DEV)
            for k in ("x", "v", "m"):
                s[k].requires_grad_(True)
        else:
            s["lam_x"], s["lam_v"] = (torch.from_numpy(rng.standard_normal((n, 3))).to(DEV) for _ in range(2))
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "forces":
        nb.nbody_forces(s["ctx"], s["x"], s["m"], s["out"]["a"], s["out"]["phi"])
        return s["out"].handed_on()
    if kind == "noalloc":
        nb.nbody_forces_noalloc(s["x"], s["m"], 1.0, case["eps"], s["out"]["a"], s["out"]["phi"])
        return s["out"].handed_on()
    if kind in ("step", "ensemble", "host"):
        call = nb.nbody_step_host if kind == "host" else nb.nbody_step
        o = s["out"]
        call(s["ctx"], o["x"], o["v"], s["m"], o["a"], True, case["steps"], o["log"] if case["every"] else None)
        return o.handed_on()
    if kind == "train":
        xT, vT = nb.NBodyAdjoint.apply(s["ctx"], s["x"], s["v"], s["m"], case["steps"], case["checkpoint"])
        loss = ((xT - s["target"]) ** 2).sum()
        g = torch.autograd.grad(loss, [s["x"], s["v"], s["m"]])
        return {k: t.float() for k, t in zip(("x", "v", "g_x", "g_v", "g_m"), (xT.detach(), vT.detach()) + g)}
    g = nb.nbody_adjoint_params(s["ctx"], s["x"], s["v"], s["m"], case["steps"], case["checkpoint"], s["lam_x"],
                                s["lam_v"])
    return dict(zip(("g_x", "g_v", "g_m", "g_params"), g))


# Floating-point operations of one unordered pair (a fused multiply-add counts two): separation and
# s^2 9, rsqrt 1, powers and the two mass factors 4, both bodies' sums 12 (+ 4 with both potentials);
# Lennard-Jones 28; the force gradient 64.
_PAIR = {"gravity": 26, "phi": 4, "lj": 28, "vjp": 64}


def work(case):
    n, kind = case["n"], case["kind"]
    sizes = [n]
    if kind == "ensemble":
        sizes = [int(k) for k in inputs.ensemble_sizes(case["systems"], case["layout"], 64, n)]
    pairs, total = sum(k * (k - 1) / 2 for k in sizes), sum(sizes)
    force = _PAIR["lj"] if case["law"] == "lj" else _PAIR["gravity"]
    if kind in ("forces", "noalloc"):
        return {"bytes": 64 * total, "flops": pairs * (force + _PAIR["phi"])}
    if kind in ("step", "ensemble", "host"):
        return {"bytes": 152 * total, "flops": pairs * case["steps"] * force}
    steps = case["steps"]
    forward = 2 * steps if kind == "train" else steps  # a stored trajectory needs each force once
    return {"bytes": 200 * total, "flops": pairs * (forward * force + (steps + 1) * _PAIR["vjp"])}


# ---- float64 results from plain torch


def _rows(n):
    k = max(1, min(n, (1 << 25) // max(1, n)))
    return [(b, min(n, b + k)) for b in range(0, n, k)]


def _pairs(x, b, e):
    """Components of d_ij = x_j - x_i for rows b..e."""
    return [x[None, :, c] - x[b:e, c, None] for c in range(3)]


def _forces64(x, m, eps, law):
    n = x.shape[0]
    a, phi = torch.empty_like(x), torch.empty_like(m)
    for b, e in _rows(n):
        d = _pairs(x, b, e)
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps
        i = torch.arange(b, e, device=x.device)
        if law == "lj":
            u = 1.0 / r2
            u[i - b, i] = 0.0
            u3 = u * u * u
            f = (u3 - 2 * u3 * u3) * u
            p = u3 * u3 - u3
            a[b:e] = torch.stack([24 * (f * c).sum(1) for c in d], 1) / m[b:e, None]
            phi[b:e] = 4 * p.sum(1) / m[b:e]
        else:
            inv = r2.rsqrt_()
            inv[i - b, i] = 0.0
            p = inv * m
            phi[b:e] = -p.sum(1)
            p *= inv
            p *= inv
            a[b:e] = torch.stack([(p * c).sum(1) for c in d], 1)
    return a, phi


def _kdk64(x, v, m, a, case, box, steps):
    """One trajectory; yields (x, v, a, phi) after each step."""
    dt = case["dt"]
    for _ in range(steps):
        v = v + 0.5 * dt * a
        x = x + dt * v
        if box > 0:
            for _ in range(4):
                low, high = x < 0, x > box
                x = torch.where(low, -x, torch.where(high, 2 * box - x, x))
                v = torch.where(low | high, -v, v)
        a, phi = _forces64(x, m, case["eps"], case["law"])
        v = v + 0.5 * dt * a
        yield x, v, a, phi


def _record64(x, v, m, phi):
    K, U = 0.5 * (m * (v * v).sum(1)).sum(), 0.5 * (m * phi).sum()
    P, L = (m[:, None] * v).sum(0), (m[:, None] * torch.linalg.cross(x, v)).sum(0)
    return torch.cat([torch.stack([K + U, K, U]), P, L])


def _vjp64(x, m, w, eps):
    """(dL/dx, dL/dm, w.da/dG, w.da/deps) of the softened force map for G = 1 and weights w = dL/da."""
    gx, gm = torch.empty_like(x), torch.empty_like(m)
    dG = de = 0.0
    for b, e in _rows(2 * x.shape[0]):
        if b >= x.shape[0]:
            break
        e = min(e, x.shape[0])
        d = _pairs(x, b, e)
        inv = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps * eps).rsqrt_()
        i = torch.arange(b, e, device=x.device)
        inv[i - b, i] = 0.0
        i3 = inv * inv * inv
        i5 = i3 * inv * inv
        wj = d[0] * w[None, :, 0] + d[1] * w[None, :, 1] + d[2] * w[None, :, 2]
        wi = d[0] * w[b:e, 0, None] + d[1] * w[b:e, 1, None] + d[2] * w[b:e, 2, None]
        t = 3 * (m[b:e, None] * wj - m[None, :] * wi) * i5
        gx[b:e] = torch.stack([(i3 * (m[b:e, None] * w[None, :, c] - m[None, :] * w[b:e, c, None]) - t * d[c]).sum(1)
                               for c in range(3)], 1)
        gm[b:e] = -(wj * i3).sum(1)
        wi *= m[None, :]
        dG = dG + (wi * i3).sum()
        de = de - 3 * eps * (wi * i5).sum()
    return gx, gm, dG, de


def _adjoint64(xs, m, lam_x, lam_v, case):
    dt, T = case["dt"], len(xs) - 1
    gm, dG, de = torch.zeros_like(m), 0.0, 0.0
    for s in range(T, -1, -1):
        coef = 0.5 * dt if s in (0, T) else dt
        gx, g, p, q = _vjp64(xs[s], m, lam_v, case["eps"])
        lam_x, gm = lam_x + coef * gx, gm + coef * g
        dG, de = dG + coef * p, de + coef * q
        if s > 0:
            lam_v = lam_v + dt * lam_x
    return lam_x, lam_v, gm, torch.stack([dG, de])[None]


def exact(case, seed):
    x, v, m, box, offsets = _bodies(case, seed)
    x, v, m = (torch.from_numpy(np.ascontiguousarray(t)).to(DEV) for t in (x, v, m))
    kind, law, eps = case["kind"], case["law"], case["eps"]
    if kind in ("forces", "noalloc"):
        a, phi = _forces64(x, m, eps, law)
        return {"a": a, "phi": phi}
    if kind in ("step", "ensemble", "host"):
        got = []
        for b, e in zip(offsets, offsets[1:]):
            ms = m[b:e]
            a, _ = _forces64(x[b:e], ms, eps, law)
            log = []
            for k, (xs, vs, a, phi) in enumerate(_kdk64(x[b:e], v[b:e], ms, a, case, box, case["steps"])):
                if case["every"] and (k + 1) % case["every"] == 0:
                    log.append(_record64(xs, vs, ms, phi))
            got.append((xs, vs, a, log))
        out = {k: torch.cat([g[i] for g in got]) for i, k in enumerate(("x", "v", "a"))}
        if case["every"]:
            out["log"] = torch.stack([torch.stack(g[3]) for g in got], 1)
        return {k: t.cpu() for k, t in out.items()} if kind == "host" else out
    a, _ = _forces64(x, m, eps, law)
    xs, vT = [x], v
    for xT, vT, a, _ in _kdk64(x, v, m, a, case, 0.0, case["steps"]):
        xs.append(xT)
    if kind == "train":
        lam_x, lam_v = 2 * (xs[-1] - torch.from_numpy(inputs.targets(len(m), seed + 1)).to(DEV)), torch.zeros_like(v)
    else:
        rng = np.random.default_rng(seed + 1)
        lam_x, lam_v = (torch.from_numpy(rng.standard_normal((len(m), 3))).to(DEV) for _ in range(2))
    g = dict(zip(("g_x", "g_v", "g_m", "g_params"), _adjoint64(xs, m, lam_x, lam_v, case)))
    if kind == "train":
        del g["g_params"]
        g.update(x=xs[-1], v=vT)
    return g
