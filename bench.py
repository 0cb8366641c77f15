#!/usr/bin/env python
"""Throughput benchmark of the N-body hot path on GB300.

Workload (one "step" = one KDK leapfrog step of the whole hot path: staging,
all-pairs mixed-precision force with fused potential, kicks and drift, float64
energy / momentum reduction): a seeded Plummer sphere of N = 65 536 bodies,
G = 1, eps = 0.005, dt = 5e-4, masses 1/N. Metric: body-body interactions per
second (N^2 per force evaluation). Beside it: the plain FP64 GPU path on the
same state, the force error of the mixed path against the FP64 CPU oracle on
sampled bodies, the force kernel's fraction of the FP32-pipe roofline, an
end-to-end figure through the host-memory entry point, and the oracle itself
timed on this host's cores.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Under torchrun every rank runs an independent system (weak scaling, no
collective on the data path); rank 0 prints one JSON line.
"""

from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "body-body interactions/s, mixed vs FP64 path at ≤1e-4 force err; % FP32 roofline"
UNIT = "interactions/s"
WORKLOAD = dict(n=65536, G=1.0, eps=0.005, dt=5e-4, seed=2)


def ops_per_interaction(sym, law="gravity", equal_masses=True, record=True):
    """float32-pipe operations per interaction in the mixed force kernels (MUFU not counted).

    One-sided: 3 FADD (d) + 3 FFMA (s^2) + 3 FMUL (m/s, 1/s^2, m/s^3) + 3 FFMA (a) + 1 FADD (phi);
    Lennard-Jones 16. Symmetric pass, per unordered pair (two interactions): 3 FADD + 3 FFMA + 2 FMUL
    (1/s^2, 1/s^3) + 2 FMUL (the masses, unless all are equal) + 6 FFMA (both bodies' forces), one more
    for an energy record; Lennard-Jones 17 and two more."""
    if law == "lj":
        return (17 + 2 * record) / 2 if sym else 14 + 2 * record
    return (14 + 2 * (not equal_masses) + record) / 2 if sym else 12 + record


def is_symmetric(nb, ctx):
    return nb.nbody_get_slicing(ctx)["tail"] >= 2


FP32_LANES_PER_SM = 128
SM_MAX_MHZ = 2070.0
L2_FLUSH_BYTES = 256 << 20
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "force_mixed_n65536_full.md")
# sources of the timed force kernel: its traffic figure is valid while their hash matches
FORCE_SRCS = [os.path.join(ROOT, "paper_2511_02655_gb300", "csrc", f)
              for f in ("sym_kernels.cu", "sym_common.cuh", "pair_common.cuh", "nbody_internal.h")]


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=500)
    p.add_argument("--warmup", type=int, default=5)
    p.add_argument("--impl", choices=("ours", "reference"), default="ours")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--no-aux", action="store_true", help="skip the other workloads' short measurements")
    p.add_argument("--aux-only", choices=("two_spheres", "ensemble", "lj", "adjoint"),
                   help="run only this one of the other workloads' measurements and print it (for profiling)")
    return p.parse_args()


def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def reduce_max(value, dist=None, device=None):
    """Max of a float over all ranks (identity without a process group)."""
    if dist is None:
        return float(value)
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank, world, max_seconds):
    """Whole-job throughput: units all ranks processed / the slowest rank's time."""
    return world * float(units_per_rank) / max_seconds


class ClockSampler:
    """nvidia-smi clock / throttle sampling while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        # raw samples: BENCH_CLOCKS_DIR if set (to keep them), else the system temp directory
        out_dir = os.environ.get("BENCH_CLOCKS_DIR") or tempfile.gettempdir()
        self.path = os.path.join(out_dir, f"clocks_bench_{os.getpid()}.csv")

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
            time.sleep(0.3)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.2)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        sm, smax, reasons = [], [], set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for line in open(self.path):
            parts = [s.strip() for s in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "reasons": sorted(reasons),
                "samples": len(sm)}


def traffic_per_launch():
    """DRAM bytes per force launch from the committed ncu summary, if it still matches the sources."""
    try:
        text = open(TRAFFIC_FILE).read()
        nbytes = re.search(r"DRAM bytes per launch \(.*?\): (\d+)", text)
        src_sha = re.search(r"Kernel source SHA-256 \(.*?\): ([0-9a-f]{64})", text)
        h = hashlib.sha256()
        for f in FORCE_SRCS:
            h.update(open(f, "rb").read())
        sha = h.hexdigest()
        if not nbytes or not src_sha or src_sha.group(1) != sha:
            return None
        return float(nbytes.group(1))
    except Exception:
        return None


def fp32_peak_tops():
    """FP32-pipe peak in T ops/s: SMs x 128 lanes x the maximum SM clock."""
    import torch
    sms = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
    return sms * FP32_LANES_PER_SM * SM_MAX_MHZ * 1e6 / 1e12


def rel_force_error(a, a_ref, guard=1e-3):
    """|a - a_ref| / |a_ref| per body, floored at guard * rms(|a_ref|) (cancellation guard)."""
    import numpy as np
    nrm = np.linalg.norm(a_ref, axis=1)
    rms = float(np.sqrt(np.mean(nrm ** 2)))
    return np.linalg.norm(a - a_ref, axis=1) / np.maximum(nrm, guard * rms)


def cpu_baseline(x, m, G, eps, a_gpu, budget_s=12.0):
    """The oracle (as it stands) on a bounded sample: forces of k seeded bodies against all N."""
    import numpy as np

    import oracle
    from paper_2511_02655_gb300 import inputs
    n = len(m)
    threads = oracle.default_threads()
    probe = inputs.sample_indices(n, 128, seed=99)
    t0 = time.perf_counter()
    oracle.forces_at(x, m, probe, G=G, eps=eps, threads=threads)
    per_body = (time.perf_counter() - t0) / len(probe)
    k = int(max(256, min(n, budget_s / max(per_body, 1e-9))))
    idx = inputs.sample_indices(n, k, seed=7)
    t0 = time.perf_counter()
    a_ref, _ = oracle.forces_at(x, m, idx, G=G, eps=eps, threads=threads)
    dt = time.perf_counter() - t0
    err = rel_force_error(a_gpu[idx], a_ref)
    # the same oracle on one host thread, on a smaller sample (about 2 s)
    k1 = int(max(16, min(n, 2.0 / max(per_body * threads, 1e-9))))
    idx1 = inputs.sample_indices(n, k1, seed=8)
    t0 = time.perf_counter()
    oracle.forces_at(x, m, idx1, G=G, eps=eps, threads=1)
    dt1 = time.perf_counter() - t0
    base = {"value": k * n / dt, "unit": UNIT, "cores": threads, "kind": "oracle",
            "sample": f"FP64 direct-sum forces of {k} seeded bodies against all {n} (1 force pass, "
                      f"{k * n:.3e} interactions, {dt:.1f} s)",
            "one_thread": {"value": k1 * n / dt1, "sample": f"{k1} seeded bodies against all {n}, {dt1:.1f} s"}}
    return base, {"median": float(np.median(err)), "max": float(err.max()), "bodies": int(k)}


def energy_vs_oracle(nb, dev, x, v, m, G, eps, dt, xf, vf, E_final, steps=3):
    """The mixed path's energy of the bench's final state against the oracle's pair-sum energy of the
    same state, and the energy drift over the first `steps` KDK steps from the initial state of the
    mixed and FP64 GPU paths beside the oracle's own KDK run."""
    import numpy as np
    import torch

    import oracle
    threads = oracle.default_threads()
    E_or_final = oracle.energy(xf, vf, m, G=G, eps=eps, threads=threads)[0]
    E_or0 = oracle.energy(x, v, m, G=G, eps=eps, threads=threads)[0]
    _, _, _, log_or = oracle.kdk(x, v, m, G, eps, dt, steps, energy_every=1, threads=threads)
    out = {"final_state_rel_err": abs(E_final - E_or_final) / abs(E_or_final),
           f"drift_first_{steps}_steps": {"oracle": float(np.abs(log_or[:, 0] - E_or0).max() / abs(E_or0))},
           f"err_vs_oracle_first_{steps}_steps": {}}
    for prec, name in ((nb.MIXED, "gpu_mixed"), (nb.FP64, "gpu_fp64")):
        c = nb.nbody_init(G=G, eps=eps, dt=dt, precision=prec, n=len(m), energy_every=1)
        xs, vs, ms = (torch.from_numpy(t).to(dev) for t in (x, v, m))
        E0 = nb.nbody_energy(c, xs, vs, ms).cpu().numpy()[0, 0]
        lg = nb.nbody_step(c, xs, vs, ms, torch.empty_like(xs), False, steps).cpu().numpy()[:, 0, 0]
        nb.nbody_sync(c)
        c.close()
        out[f"drift_first_{steps}_steps"][name] = float(np.abs(lg - E0).max() / abs(E0))
        out[f"err_vs_oracle_first_{steps}_steps"][name] = float(np.abs(lg - log_or[:, 0]).max() / abs(E_or0))
    return out


def _event_time(fn, stream, nvtx=None):
    """CUDA-event seconds of fn() on stream; the launches sit in NVTX range `nvtx` (for ncu filters)."""
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    if nvtx:
        torch.cuda.nvtx.range_push(nvtx)
    e0.record(stream)
    fn()
    e1.record(stream)
    if nvtx:
        torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) * 1e-3


def _err_stats(err):
    import numpy as np
    err = np.asarray(err)
    return {"median": float(np.median(err)), "max": float(err.max()), "n": int(err.size)}


def _elem_err(g, g_ref, guard=1e-3):
    """Per-element relative error, floored at guard * rms(g_ref) (cancellation guard)."""
    import numpy as np
    g, g_ref = np.asarray(g).ravel(), np.asarray(g_ref).ravel()
    rms = float(np.sqrt(np.mean(g_ref ** 2)))
    return np.abs(g - g_ref) / np.maximum(np.abs(g_ref), guard * rms)


def _timed(fn):
    t0 = time.perf_counter()
    out = fn()
    return out, time.perf_counter() - t0


def aux_two_spheres(dev, stream):
    """Two Plummer spheres, N = 1 048 576, eps = 0.002, dt = 5e-4, mixed: throughput, force error
    against the oracle on 16 384 sampled bodies at the start and after the timed steps, energy drift,
    and the oracle's rate on those samples extrapolated to a whole force pass."""
    import numpy as np
    import torch

    import oracle
    import paper_2511_02655_gb300 as nb
    from paper_2511_02655_gb300 import inputs
    n, G, eps, dt, k, ks = 1048576, 1.0, 0.002, 5e-4, 3, 16384
    x, v, m = inputs.two_spheres(n, seed=3)
    ctx = nb.nbody_init(G=G, eps=eps, dt=dt, precision=nb.MIXED, n=n)
    xt, vt, mt = (torch.from_numpy(t).to(dev) for t in (x, v, m))
    at = torch.empty_like(xt)
    nb.nbody_forces(ctx, xt, mt, at, None, with_phi=False)
    a0 = at.cpu().numpy()
    E0 = nb.nbody_energy(ctx, xt, vt, mt).cpu().numpy()[0, 0]
    nb.nbody_profile(ctx, True)
    sec = _event_time(lambda: nb.nbody_step(ctx, xt, vt, mt, at, True, k), stream, "aux_two_spheres")
    kms, kl = nb.nbody_kernel_time(ctx, 0)
    nb.nbody_profile(ctx, False)
    E1 = nb.nbody_energy(ctx, xt, vt, mt).cpu().numpy()[0, 0]
    nb.nbody_sync(ctx)
    xf, af = xt.cpu().numpy(), at.cpu().numpy()
    tuning = nb.nbody_get_tuning(ctx)
    ops = ops_per_interaction(is_symmetric(nb, ctx), equal_masses=False, record=False)
    ctx.close()
    del xt, vt, mt, at
    threads = oracle.default_threads()
    idx0, idx1 = inputs.sample_indices(n, ks, seed=17), inputs.sample_indices(n, ks, seed=19)
    (ref0, _), t0 = _timed(lambda: oracle.forces_at(x, m, idx0, G=G, eps=eps, threads=threads))
    (ref1, _), t1 = _timed(lambda: oracle.forces_at(xf, m, idx1, G=G, eps=eps, threads=threads))
    rate = 2.0 * ks * n / (t0 + t1)
    return {"interactions_per_s": float(n) * n * k / sec, "steps": k, "force_kernel_ms": kms / kl,
            "frac_fp32_roofline_force_kernel": ops * float(n) * n / (kms / kl * 1e-3) / 1e12
                                               / fp32_peak_tops(),
            "tuning": tuning,
            "force_err_vs_oracle": {"step_0": _err_stats(rel_force_error(a0[idx0], ref0)),
                                    f"step_{k}": _err_stats(rel_force_error(af[idx1], ref1)),
                                    "sample": f"{ks} seeded bodies against all {n}, FP64 oracle"},
            "energy_drift_rel": float(abs(E1 - E0) / abs(E0)),
            "cpu_baseline": {"value": rate, "unit": UNIT, "cores": threads, "kind": "oracle",
                             "sample": f"FP64 forces of 2 x {ks} seeded bodies against all {n} (the error samples), "
                                       f"{t0 + t1:.1f} s",
                             "extrapolated_s_per_force_pass": float(n) * n / rate,
                             "extrapolation": "extrapolated by N^2 from the sampled rows"}}


def aux_ensemble(dev, stream):
    """512 Plummer systems, N log-uniform in [64, 16384], eps = 0.01, dt = 1e-3, 50 steps per call in one
    persistent launch per step replayed as a CUDA graph, beside 512 per-system FP64 launch sequences;
    per-system sampled force error and energy drift; the oracle on a seeded subset of whole systems,
    extrapolated by sum N^2."""
    import numpy as np
    import torch

    import oracle
    import paper_2511_02655_gb300 as nb
    from paper_2511_02655_gb300 import inputs
    G, eps, dt, T = 1.0, 0.01, 1e-3, 50
    ens = inputs.ensemble(512, seed=4)
    off = [int(o) for o in ens.offsets]
    sizes = np.diff(ens.offsets).astype(np.int64)
    pairs = float((sizes.astype(np.float64) ** 2).sum())
    ctx = nb.nbody_init(G=G, eps=eps, dt=dt, precision=nb.MIXED, offsets=off, energy_every=T, flags=nb.FLAG_GRAPH)
    xt, vt, mt = (torch.from_numpy(t).to(dev) for t in (ens.x, ens.v, ens.m))
    at = torch.empty_like(xt)
    log = torch.empty((1, 512, 9), dtype=torch.float64, device=dev)
    nb.nbody_forces(ctx, xt, mt, at, None, with_phi=False)
    nb.nbody_step(ctx, xt, vt, mt, at, True, T, log)  # captures the graph
    E0 = nb.nbody_energy(ctx, xt, vt, mt).cpu().numpy()[:, 0]
    l0 = nb.nbody_launch_count(ctx)
    sec = _event_time(lambda: nb.nbody_step(ctx, xt, vt, mt, at, True, T, log), stream, "aux_ensemble")
    nb.nbody_sync(ctx)
    launches = nb.nbody_launch_count(ctx) - l0
    E1 = log.cpu().numpy()[0, :, 0]
    xf, af = xt.cpu().numpy(), at.cpu().numpy()
    ctx.close()
    # the same systems as 512 separate FP64 contexts, one launch sequence per system, 1 step
    ctxs, bufs = [], []
    for s_ in range(512):
        b, e = off[s_], off[s_ + 1]
        c1 = nb.nbody_init(G=G, eps=eps, dt=dt, precision=nb.FP64, n=e - b, block=128, i_per_thread=1, j_tile=128)
        xs, vs, ms = (torch.from_numpy(np.ascontiguousarray(t[b:e])).to(dev) for t in (ens.x, ens.v, ens.m))
        a1 = torch.empty_like(xs)
        nb.nbody_forces(c1, xs, ms, a1, None, with_phi=False)
        ctxs.append(c1), bufs.append((xs, vs, ms, a1))

    def per_system():
        for c1, (xs, vs, ms, a1) in zip(ctxs, bufs):
            nb.nbody_step(c1, xs, vs, ms, a1, True, 1)

    sec64 = _event_time(per_system, stream, "aux_ensemble_fp64")
    for c1 in ctxs:
        c1.close()
    # force error at the final state: up to 32 seeded bodies of every system against its own bodies
    errs, worst = [], 0.0
    for s_ in range(512):
        b, e = off[s_], off[s_ + 1]
        idx = inputs.sample_indices(e - b, min(32, e - b), seed=1000 + s_)
        ref, _ = oracle.forces_at(xf[b:e], ens.m[b:e], idx, G=G, eps=eps, threads=1)
        err = rel_force_error(af[b:e][idx], ref)
        errs.append(err)
        worst = max(worst, float(err.max()))
    # the oracle on 16 seeded whole systems (one force pass each), extrapolated by sum N^2
    threads = oracle.default_threads()
    sel = np.random.default_rng(77).choice(512, 16, replace=False)
    _, t_or = _timed(lambda: [oracle.forces(ens.x[off[s_]:off[s_ + 1]], ens.m[off[s_]:off[s_ + 1]], G=G, eps=eps,
                                            threads=threads, with_phi=False) for s_ in sel])
    sub_pairs = float((sizes[sel].astype(np.float64) ** 2).sum())
    rate = sub_pairs / t_or
    drift = np.abs(E1 - E0) / np.abs(E0)
    return {"mixed_graph_interactions_per_s": pairs * T / sec, "steps": T,
            "fp64_per_system_interactions_per_s": pairs / sec64,
            "graph_over_fp64_per_system": (pairs * T / sec) / (pairs / sec64),
            "pairs_per_step": pairs, "launches_per_50_steps": int(launches),
            "force_err_vs_oracle": dict(_err_stats(np.concatenate(errs)), worst_system_max=worst,
                                        sample="final state, up to 32 seeded bodies of each of the 512 systems "
                                               "against that system, FP64 oracle"),
            "energy_drift_rel_over_50_steps": {"max": float(drift.max()), "median": float(np.median(drift))},
            "cpu_baseline": {"value": rate, "unit": UNIT, "cores": threads, "kind": "oracle",
                             "sample": f"FP64 force pass of 16 seeded whole systems ({sub_pairs:.3e} interactions, "
                                       f"{t_or:.2f} s)",
                             "extrapolated_s_per_step": pairs / rate,
                             "extrapolation": "extrapolated by sum N^2 over the 512 systems"}}


def aux_lj(dev, stream):
    """The paper's own system: Lennard-Jones gas, 10 000 particles, 2500 KDK steps with the total energy
    reduced every step, reflecting walls (reduced units, density 0.05, T = 2, dt = 5e-3); sampled force
    error at the end, energy drift beside the oracle's over the first 20 steps, and the oracle's time for
    those 20 steps extrapolated to the whole run."""
    import numpy as np
    import torch

    import oracle
    import paper_2511_02655_gb300 as nb
    from paper_2511_02655_gb300 import inputs
    n, steps, dt, k20 = 10000, 2500, 5e-3, 20
    x, v, m, box = inputs.lj_gas(n, seed=9)
    E_or0 = oracle.lj_energy(x, v, m)[0]
    threads = oracle.default_threads()
    (_, _, _, log_or), t_or = _timed(lambda: oracle.lj_kdk(x, v, m, 1.0, 1.0, 0.0, box, dt, k20, energy_every=1,
                                                           threads=threads))
    lj = {}
    for prec, flags, name in ((nb.MIXED, nb.FLAG_GRAPH, "mixed_graph"), (nb.FP64, 0, "fp64")):
        ctx = nb.nbody_init(law=nb.LENNARD_JONES, precision=prec, n=n, dt=dt, box=box, energy_every=1,
                            flags=flags)
        xt, vt, mt = (torch.from_numpy(a).to(dev) for a in (x, v, m))
        at = torch.empty_like(xt)
        logt = torch.empty((steps, 1, 9), dtype=torch.float64, device=dev)
        E_gpu0 = nb.nbody_energy(ctx, xt, vt, mt).cpu().numpy()[0, 0]
        if flags:  # capture once on a copy of the state, replay on the real one
            x2, v2, a2 = xt.clone(), vt.clone(), torch.empty_like(xt)
            nb.nbody_step(ctx, x2, v2, mt, a2, False, steps, logt)
            nb.nbody_sync(ctx)
            x2.copy_(xt), v2.copy_(vt)
            xt, vt, at = x2, v2, a2
        sec = _event_time(lambda: nb.nbody_step(ctx, xt, vt, mt, at, False, steps, logt), stream, f"aux_lj_{name}")
        nb.nbody_sync(ctx)
        kernel = None
        if prec == nb.MIXED:  # the force kernel alone: CUDA events around it in 200 eagerly issued steps
            ce = nb.nbody_init(law=nb.LENNARD_JONES, precision=prec, n=n, dt=dt, box=box, energy_every=1)
            tun = nb.nbody_get_tuning(ce)
            ops = ops_per_interaction(is_symmetric(nb, ce), law="lj")
            xe, ve, ae = (torch.from_numpy(a).to(dev) for a in (x, v, np.zeros_like(x)))
            le = torch.empty((200, 1, 9), dtype=torch.float64, device=dev)
            nb.nbody_step(ce, xe, ve, mt, ae, False, 20, le[:20])
            nb.nbody_profile(ce, True)
            eager = _event_time(lambda: nb.nbody_step(ce, xe, ve, mt, ae, True, 200, le), stream, "aux_lj_mixed_eager")
            ms, k = nb.nbody_kernel_time(ce, 0)
            nb.nbody_profile(ce, False)
            nb.nbody_sync(ce)
            ce.close()
            us = ms * 1e3 / max(1, k)
            kernel = {"tuning": tun, "force_kernel_us": us, "eager_step_us": eager / 200 * 1e6,
                      "ops_per_interaction": ops,
                      "frac_fp32_roofline_force_kernel": ops * n * n / (us * 1e-6) / (fp32_peak_tops() * 1e12)}
        e = logt.cpu().numpy()[:, 0, 0]
        xf, af = xt.cpu().numpy(), at.cpu().numpy()
        idx = inputs.sample_indices(n, 2048, seed=29)
        ref, _ = oracle.lj_forces_at(xf, m, idx, threads=threads)
        lj[name] = {"seconds": sec, "interactions_per_s": float(n) * n * (steps + 1) / sec,
                    "energy_drift_max_rel": float(np.abs(e - E_gpu0).max() / abs(E_gpu0)),
                    "energy_drift_first_20_steps": float(np.abs(e[:k20] - E_gpu0).max() / abs(E_gpu0)),
                    "energy_err_vs_oracle_first_20_steps": float(np.abs(e[:k20] - log_or[:, 0]).max() / abs(E_or0)),
                    "force_err_vs_oracle_at_end": dict(_err_stats(rel_force_error(af[idx], ref)),
                                                       sample="2048 seeded particles after 2500 steps, FP64 oracle")}
        if kernel:
            lj[name]["force_kernel"] = kernel
        ctx.close()
    return dict(lj, oracle_energy_drift_first_20_steps=float(np.abs(log_or[:, 0] - E_or0).max() / abs(E_or0)),
                cpu_baseline={"value": float(n) * n * (k20 + 1) / t_or, "unit": UNIT, "cores": threads,
                              "kind": "oracle", "sample": f"the FP64 oracle's KDK run of the first {k20} steps "
                                                          f"with the energy every step, {t_or:.1f} s",
                              "extrapolated_s_for_2500_steps": t_or * steps / k20,
                              "extrapolation": "extrapolated by the step count"},
                context="paper (Sec. VI): 19.02 s median, RAJA, 4x A100, FP64, with energy reduction; other "
                        "hardware, context only")


def aux_adjoint(dev, stream):
    """Adjoint: N = 16384 Plummer, 200 KDK steps, dt = 1e-3, checkpoints every 20, loss sum |x_T - t|^2.
    Times both precisions; the mixed gradients per element against the FP64 ones; both against FP64
    central differences (h = 1e-6) of the FP64 GPU trajectory on 3 seeded coordinates; and the CPU
    reference adjoint (the oracle) at N = 2048, timed and compared with the GPU adjoints there."""
    import numpy as np
    import torch

    import oracle
    import paper_2511_02655_gb300 as nb
    from paper_2511_02655_gb300 import inputs
    G, eps, dt, T, K = 1.0, 0.01, 1e-3, 200, 20
    out, grads = {}, {}

    def final_lam(n):
        """dL/dx_T = 2 (x_T - t) from the FP64 GPU trajectory (shared by both precisions' adjoints, so
        that their gradients differ only by the adjoint's own arithmetic)."""
        x, v, m = inputs.plummer(n, seed=5)
        t = torch.from_numpy(inputs.targets(n, seed=6)).to(dev)
        ctx = nb.nbody_init(G=G, eps=eps, dt=dt, precision=nb.FP64, n=n)
        xs, vs, mt = (torch.from_numpy(a).to(dev) for a in (x, v, m))
        nb.nbody_step(ctx, xs, vs, mt, torch.empty_like(xs), False, T)
        nb.nbody_sync(ctx)
        ctx.close()
        return 2 * (xs - t)

    def run(n, prec, lam, timed_name=None):
        x, v, m = inputs.plummer(n, seed=5)
        ctx = nb.nbody_init(G=G, eps=eps, dt=dt, precision=prec, n=n)
        xt, vt, mt = (torch.from_numpy(a).to(dev) for a in (x, v, m))
        zero = torch.zeros_like(xt)
        g = nb.nbody_adjoint(ctx, xt, vt, mt, T, K, lam, zero)  # tunes the VJP tiling
        sec = None
        if timed_name:
            sec = _event_time(lambda: nb.nbody_adjoint(ctx, xt, vt, mt, T, K, lam, zero, *g), stream,
                              f"aux_{timed_name}")
        nb.nbody_sync(ctx)
        ctx.close()
        return sec, [a.cpu().numpy() for a in g]

    n = 16384
    lam = final_lam(n)
    for prec, name in ((nb.MIXED, "adjoint_16384_mixed"), (nb.FP64, "adjoint_16384_fp64")):
        sec, grads[prec] = run(n, prec, lam, name)
        out[name] = {"seconds": sec, "steps": T, "checkpoint_every": K,
                     "force_passes": T + 1 + (T // K - 1) * (K - 1), "vjp_passes": T + 1}
    out["adjoint_16384_mixed"]["grad_err_vs_fp64_gpu"] = {  # same dL/dx_T for both
        nm: _err_stats(_elem_err(gm, g64)) for nm, gm, g64 in zip(("x0", "v0", "m"), grads[nb.MIXED], grads[nb.FP64])}
    # central differences on the FP64 GPU path: one position, one velocity and one mass coordinate
    x, v, m = inputs.plummer(n, seed=5)
    t = torch.from_numpy(inputs.targets(n, seed=6)).to(dev)
    rng = np.random.default_rng(7)
    i_x, c_x, i_v, c_v, i_m = (int(rng.integers(n)), int(rng.integers(3)), int(rng.integers(n)), int(rng.integers(3)),
                               int(rng.integers(n)))
    h, copies = 1e-6, []
    for sgn in (1.0, -1.0):
        for kind in ("x", "v", "m"):
            xx, vv, mm = x.copy(), v.copy(), m.copy()
            if kind == "x":
                xx[i_x, c_x] += sgn * h
            elif kind == "v":
                vv[i_v, c_v] += sgn * h
            else:
                mm[i_m] += sgn * h
            copies.append((xx, vv, mm))
    offs = [k_ * n for k_ in range(7)]
    ctxb = nb.nbody_init(G=G, eps=eps, dt=dt, precision=nb.FP64, offsets=offs)
    xb, vb, mb = (torch.from_numpy(np.concatenate([c[j] for c in copies])).to(dev) for j in range(3))
    nb.nbody_step(ctxb, xb, vb, mb, torch.empty_like(xb), False, T)
    nb.nbody_sync(ctxb)
    ctxb.close()
    xr = xb.view(6, n, 3)
    dL = ((xr[0:3] - xr[3:6]) * (xr[0:3] + xr[3:6] - 2 * t)).sum(dim=(1, 2)).cpu().numpy()
    fd = dL / (2 * h)
    for prec, name in ((nb.MIXED, "adjoint_16384_mixed"), (nb.FP64, "adjoint_16384_fp64")):
        gx, gv, gm = grads[prec]
        ad = np.array([gx[i_x, c_x], gv[i_v, c_v], gm[i_m]])
        out[name]["grad_err_vs_central_differences"] = {
            "max": float((np.abs(ad - fd) / np.abs(fd)).max()), "coordinates": 3,
            "note": "x, v and m coordinates of seeded bodies; FP64 GPU trajectories, h = 1e-6"}
    # CPU reference adjoint (the oracle) at reduced N, beside the GPU adjoints at that N
    n2 = 2048
    x2, v2, m2 = inputs.plummer(n2, seed=5)
    threads = oracle.default_threads()
    lam2 = final_lam(n2)
    _, g_mixed = run(n2, nb.MIXED, lam2)
    _, g_fp64 = run(n2, nb.FP64, lam2)
    lam2 = lam2.cpu().numpy()
    (gref), t_or = _timed(lambda: oracle.adjoint(x2, v2, m2, G, eps, dt, T, lam2, np.zeros_like(lam2),
                                                 threads=threads))
    out["adjoint_reduced_n2048"] = {
        "grad_err_vs_oracle": {
            pname: {nm: _err_stats(_elem_err(g, r)) for nm, g, r in zip(("x0", "v0", "m"), gg, gref)}
            for pname, gg in (("mixed", g_mixed), ("fp64", g_fp64))},
        "cpu_baseline": {"value": t_or, "unit": "s", "cores": threads, "kind": "oracle",
                         "sample": f"the CPU reference adjoint (full trajectory stored, FP64) at N = {n2}, {T} steps",
                         "extrapolated_s_at_n16384": t_or * (16384 / n2) ** 2,
                         "extrapolation": "extrapolated by N^2 from the reduced N"}}
    return out


def aux_measurements(dev):
    """The other workloads, each measured briefly (rank 0, one GPU): CUDA-event times around
    nbody_step / nbody_adjoint calls, initialisation and autotuning excluded; beside each throughput
    its error against the FP64 oracle and the oracle's own (sampled, extrapolated) time."""
    import torch
    stream = torch.cuda.current_stream()
    out = {"two_spheres_1m": aux_two_spheres(dev, stream)}
    out["ensemble_512"] = aux_ensemble(dev, stream)
    out["paper_lj_gas_10000x2500"] = aux_lj(dev, stream)
    out.update(aux_adjoint(dev, stream))
    return out


def run_aux_only(args):
    """One of the other workloads' measurements alone (rank 0, one GPU), printed as one JSON line."""
    import torch
    import paper_2511_02655_gb300 as nb
    rank, world, local = dist_env()
    if rank != 0:
        return 0
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    nb.load()
    stream = torch.cuda.current_stream()
    fn = {"two_spheres": aux_two_spheres, "ensemble": aux_ensemble, "lj": aux_lj}.get(args.aux_only)
    out = fn(dev, stream) if fn else aux_adjoint(dev, stream)
    print(json.dumps({"aux_only": args.aux_only, "result": out}), flush=True)
    return 0


def run_reference(args):
    """The CPU oracle on this host's cores, on the same workload: each step is a bounded sample."""
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    import oracle
    from paper_2511_02655_gb300 import inputs
    w = WORKLOAD
    x, v, m = inputs.plummer(w["n"], seed=w["seed"])
    n = w["n"]
    threads = oracle.default_threads()
    probe = inputs.sample_indices(n, 64, seed=98)
    t0 = time.perf_counter()
    oracle.forces_at(x, m, probe, G=w["G"], eps=w["eps"], threads=threads)
    per_body = (time.perf_counter() - t0) / len(probe)
    per_step_budget = max(0.05, 150.0 / max(1, args.steps + args.warmup))
    k = int(max(32, min(n, per_step_budget / max(per_body, 1e-9))))
    for s in range(args.warmup):
        oracle.forces_at(x, m, inputs.sample_indices(n, k, seed=1000 + s), G=w["G"], eps=w["eps"], threads=threads)
    t0 = time.perf_counter()
    for s in range(args.steps):
        oracle.forces_at(x, m, inputs.sample_indices(n, k, seed=2000 + s), G=w["G"], eps=w["eps"], threads=threads)
    dt = time.perf_counter() - t0
    value = k * n * args.steps / dt
    sample = f"each step: FP64 direct-sum forces of {k} seeded bodies against all {n}"
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt / args.steps * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": "plummer N=65536 eps=0.005 (CPU oracle, sampled rows)",
                                             "n_bodies": n, "sample_bodies_per_step": k},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": threads, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)
    return 0


def run_ours(args):
    import numpy as np
    import torch

    import paper_2511_02655_gb300 as nb
    from paper_2511_02655_gb300 import inputs

    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    pg = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
        pg = dist
    nb.load()  # fails loudly without the built library
    w = WORKLOAD
    n, G, eps, dt = w["n"], w["G"], w["eps"], w["dt"]
    x, v, m = inputs.plummer(n, seed=w["seed"] + rank)
    K, W = args.steps, max(3, args.warmup)
    stream = torch.cuda.current_stream()

    # ---- mixed path: init + autotune (excluded from timing, as the paper excludes initialisation)
    ctx = nb.nbody_init(G=G, eps=eps, dt=dt, precision=nb.MIXED, n=n, energy_every=1)
    tuning = nb.nbody_get_tuning(ctx)
    xt, vt, mt = (torch.from_numpy(t).to(dev) for t in (x, v, m))
    at = torch.empty_like(xt)
    nb.nbody_forces(ctx, xt, mt, at, None, with_phi=False)
    a0 = at.cpu().numpy()
    E0 = nb.nbody_energy(ctx, xt, vt, mt).cpu().numpy()[0, 0]
    log = torch.empty((W + K, 1, 9), dtype=torch.float64, device=dev)
    for k in range(W):
        nb.nbody_step(ctx, xt, vt, mt, at, True, 1, log[k:k + 1])
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
    torch.cuda.synchronize()
    if pg:
        pg.barrier()
    clocks = ClockSampler(local)
    clocks.start()
    launches0 = nb.nbody_launch_count(ctx)
    nb.nbody_profile(ctx, True)
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_push("bench_timed")  # lets ncu select the timed launches (--nvtx-include)
    for k in range(K):
        flush.zero_()  # L2 flush between timed steps (outside the events)
        ev[k][0].record(stream)
        nb.nbody_step(ctx, xt, vt, mt, at, True, 1, log[W + k:W + k + 1])
        ev[k][1].record(stream)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    if pg:
        pg.barrier()
    clk = clocks.stop()
    launches = nb.nbody_launch_count(ctx) - launches0
    force_ms, force_launches = nb.nbody_kernel_time(ctx, 0)
    nb.nbody_profile(ctx, False)
    nb.nbody_sync(ctx)
    total_ms = reduce_max(sum(a.elapsed_time(b) for a, b in ev), pg, dev)
    interactions = float(n) * n
    value = whole_job_rate(interactions * K, world, total_ms * 1e-3)
    elog = log.cpu().numpy()[:, 0, 0]
    drift = float(np.abs(elog - E0).max() / abs(E0))

    # ---- dominant kernel vs its roofline (FP32 pipe, derived from SM count and max clock): the force
    # kernel of the timed steps (with the potential: every step records its energy)
    kernel_s = force_ms * 1e-3 / max(1, force_launches)
    sym = is_symmetric(nb, ctx)
    ops = ops_per_interaction(sym)
    achieved = ops * interactions / kernel_s / 1e12
    peak = fp32_peak_tops()
    traffic = traffic_per_launch()

    # ---- plain FP64 GPU path on the same state (a few steps)
    ctx64 = nb.nbody_init(G=G, eps=eps, dt=dt, precision=nb.FP64, n=n)
    x64, v64, a64 = xt.clone(), vt.clone(), torch.empty_like(xt)
    nb.nbody_forces(ctx64, x64, mt, a64, None, with_phi=False)
    nb.nbody_step(ctx64, x64, v64, mt, a64, True, 1)
    k64 = 3
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_push("fp64_path")
    e0.record(stream)
    nb.nbody_step(ctx64, x64, v64, mt, a64, True, k64)
    e1.record(stream)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    fp64_value = interactions * k64 / (e0.elapsed_time(e1) * 1e-3)
    ctx64.close()

    # ---- end to end through the host-memory entry point (pinned buffers, copies inside the timing):
    # a context of its own tuning that replays its step as a CUDA graph; L2 flushed between
    # steps outside the timing, each call timed on the host clock (it returns after its sync)
    ke = max(3, min(K, 50))
    ctx_h = nb.nbody_init(G=G, eps=eps, dt=dt, precision=nb.MIXED, n=n, energy_every=1, flags=nb.FLAG_GRAPH)
    xh = xt.cpu().pin_memory()
    vh = vt.cpu().pin_memory()
    mh = mt.cpu().pin_memory()
    ah = at.cpu().pin_memory()
    lh = torch.empty((1, 1, 9), dtype=torch.float64).pin_memory()
    for _ in range(W):
        nb.nbody_step_host(ctx_h, xh, vh, mh, ah, True, 1, lh)
    e2e_s = 0.0
    for _ in range(ke):
        flush.fill_(1)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        nb.nbody_step_host(ctx_h, xh, vh, mh, ah, True, 1, lh)
        e2e_s += time.perf_counter() - t0
    e2e_s = reduce_max(e2e_s, pg, dev)
    ctx_h.close()
    e2e = {"value": whole_job_rate(interactions * ke, world, e2e_s), "unit": UNIT,
           "h2d_bytes_per_step": n * 10 * 8, "d2h_bytes_per_step": n * 9 * 8 + 9 * 8,
           "call": "nbody_step_host (1 KDK step per call, pinned host x, v, m, a in; x, v, a, energy out; "
                   "step replayed as a CUDA graph; L2 flushed between calls, outside the timing)"}

    # ---- CPU oracle on this host (rank 0, N = 1 only), which also gives the force error, the
    # energy error of the final state and the oracle's own energy drift beside the GPU's
    base, ferr, eerr = None, None, None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        base, ferr = cpu_baseline(x, m, G, eps, a0)
        eerr = energy_vs_oracle(nb, dev, x, v, m, G, eps, dt, xt.cpu().numpy(), vt.cpu().numpy(),
                                float(elog[-1]))
    ctx.close()
    aux = None
    if rank == 0 and world == 1 and not args.no_aux:
        del xt, vt, mt, at, flush
        torch.cuda.empty_cache()
        aux = aux_measurements(dev)

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K, "warmup": W,
            "ms_per_step": total_ms / K, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {
                "workload": "Plummer sphere N=65536 (seeded), G=1, eps=0.005, dt=5e-4, 1 KDK step + energy/"
                            "momentum reduction per step, mixed precision",
                "n_bodies": n, "precision": "f32 pair arithmetic, compensated f32 tile sums, f64 slice sums, "
                                            "f64 state and reductions",
                "l2": "flushed (256 MiB write) between timed steps",
                "tuning": tuning,
                "fp64_path_interactions_per_s": fp64_value,
                "mixed_over_fp64": value / world / fp64_value,
                "force_err_vs_oracle": ferr,
                "energy_drift_max_rel": drift,
                "energy_vs_oracle": eerr,
                "interactions_per_step": interactions,
            },
            "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "Tops/s (FP32 pipe)",
                         "frac": achieved / peak, "traffic": traffic,
                         "kernel": "k_force_sym (every unordered pair once, packed float32x2, energy record)" if sym
                                   else "k_force_mixed2 (packed float32x2 pair arithmetic with the potential)",
                         "ops_per_interaction": ops,
                         "kernel_ms": kernel_s * 1e3,
                         "peak_basis": f"{torch.cuda.get_device_properties(dev).multi_processor_count} SMs x "
                                       f"{FP32_LANES_PER_SM} FP32 lanes x {SM_MAX_MHZ:.0f} MHz"},
            "cpu_baseline": base,
            "e2e": e2e,
            "clocks": clk,
            "gpu_launches": int(launches),
            "aux": aux,
        }
        print(json.dumps(line), flush=True)
    if pg:
        pg.barrier()
        pg.destroy_process_group()
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.aux_only:
        return run_aux_only(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
