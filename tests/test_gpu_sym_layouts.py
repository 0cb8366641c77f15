"""The symmetric passes over layouts of many bodies: 128-body chunks with 64-body i-tiles."""

import numpy as np
import pytest

import oracle
from paper_2511_02655_gb300 import inputs
from helpers import assert_elem_close, elem_rel_err, force_rel_err, to_dev
from test_gpu_sym import _forced, _masses

pytestmark = pytest.mark.gpu

# Mixed gradients of 9000 and more bodies with random weights, or of widely spread masses: elements below 1e-2
# of the rms are sums that cancel to less than float32 keeps to 1e-4 (the one-sided kernels have 2e-4, 3.3e-4 and
# 1.3e-4 at a guard of 1e-3)
GUARD = 1e-2


def _lines(path, tilings):
    """Replaces the choices of the tuning cache by the given ones ({"force" | "vjp": cache line})."""
    keys = dict.fromkeys(line.split("\t")[0] for line in path.read_text().splitlines())
    path.write_text("".join(f"{k}\t{' '.join(map(str, t))}\n" for k in keys for kind, t in tilings.items()
                            if f"|{kind}|" in k))


@pytest.mark.parametrize("sizes", [[200] * 200, [256] * 512, [33000], [0, 1, 300, 40001, 2, 4097, 63]],
                         ids=["200x200", "512x256", "33000", "uneven"])
def test_sym64_rows_hold_whole_chunks(nb, tmp_path, monkeypatch, sizes):
    """Forces, potentials, energies and gradients of FP64 layouts above 32 768 bodies in i-tiles of 64."""
    import torch
    cache = tmp_path / "tune"
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(cache))
    G, eps, dt = 1.1, 0.05, 1e-3
    ens = inputs.ensemble(len(sizes), seed=9, sizes=np.array(sizes))
    off = [int(o) for o in ens.offsets]
    x, v, m = ens.x, ens.v, _masses(ens.m, "lognormal", 9)
    rng = np.random.default_rng(9)
    lx, lv = rng.standard_normal(x.shape), 0.1 * rng.standard_normal(x.shape)
    args = to_dev(x, v, m) + (1, 1) + to_dev(lx, lv)
    kw = dict(G=G, eps=eps, dt=dt, offsets=off, precision=nb.FP64)
    ctx = nb.nbody_init(**kw)
    nb.nbody_adjoint(ctx, *args)
    ctx.close()
    sample = [s for s in (0, 1, len(sizes) // 2, len(sizes) - 1, 3, 5) if s < len(sizes)]
    refs = {}
    for s in dict.fromkeys(sample):
        b, e = off[s], off[s + 1]
        if e - b > 1:
            k = slice(b, e)
            refs[s] = (oracle.forces(x[k], m[k], G=G, eps=eps), oracle.energy(x[k], v[k], m[k], G=G, eps=eps),
                       oracle.adjoint_params(x[k], v[k], m[k], G, eps, dt, 1, lx[k], lv[k]))
    for tail in (0, 1, 2):
        _lines(cache, {"force": (64, 1, 64, 100, 3, tail), "vjp": (64, 1, 64, 100, 3, tail)})
        ctx = nb.nbody_init(**kw)
        assert nb.nbody_get_slicing(ctx)["tail"] == 2 + tail
        a, phi = nb.nbody_forces(ctx, args[0], args[2])
        en = nb.nbody_energy(ctx, args[0], args[1], args[2])
        gx, gv, gm, gp = nb.nbody_adjoint_params(ctx, *args)
        nb.nbody_sync(ctx)
        ctx.close()
        for s, ((a_ref, phi_ref), e_ref, (ox, ov, om, (oG, oe))) in refs.items():
            k = slice(off[s], off[s + 1])
            # rounding of the sums grows with their terms: ten times the bounds of test_gpu_sym.py, which has 2500
            tol = 1e-12 if off[s + 1] - off[s] <= 2500 else 1e-11
            assert force_rel_err(a[k].cpu().numpy(), a_ref).max() <= tol, (tail, s)
            assert_elem_close(phi[k].cpu().numpy(), phi_ref, tol, f"phi {tail} {s}")
            np.testing.assert_allclose(en[s].cpu().numpy()[:3], np.asarray(e_ref)[:3], rtol=tol)
            for g, o, what in ((gx, ox, "g_x0"), (gv, ov, "g_v0"), (gm, om, "g_m")):
                assert_elem_close(g[k].cpu().numpy(), o, 10 * tol, f"{what} {tail} {s}")
            gG, ge = gp[s].cpu().numpy()
            scale = max(abs(oG), abs(oe) * eps)
            assert abs(gG - oG) <= 10 * tol * scale and abs(ge - oe) * eps <= 10 * tol * scale, (tail, s)


@pytest.mark.parametrize("prec,n,cap_mb,sym", [(1, 9000, 0, False), (0, 700, 0, False), (0, 2500, 3, None),
                                               (1, 9000, 8, None), (0, 2500, 64, True), (1, 9000, 64, True)])
def test_layouts_over_the_memory_cap_still_run(nb, monkeypatch, prec, n, cap_mb, sym):
    """Lists over the cap of the symmetric passes' partial sums are left out; where none is below it, the
    one-sided pass serves sizes at which it is no candidate otherwise."""
    monkeypatch.setenv("NBODY_SYM_PARTIAL_MB", str(cap_mb))
    G, eps, dt = 1.1, 0.05, 1e-3
    x, v, m = inputs.plummer(n, seed=n)
    rng = np.random.default_rng(n)
    lx, lv = rng.standard_normal((n, 3)), 0.1 * rng.standard_normal((n, 3))
    ctx = nb.nbody_init(G=G, eps=eps, dt=dt, n=n, precision=prec)
    slicing = nb.nbody_get_slicing(ctx)
    chosen = slicing["tail"] >= 2
    assert sym is None or chosen == sym
    assert not chosen or slicing["max_slices"] * n * 32 <= cap_mb << 20
    a, phi = nb.nbody_forces(ctx, *to_dev(x, m))
    got = nb.nbody_adjoint(ctx, *to_dev(x, v, m), 1, 1, *to_dev(lx, lv))
    nb.nbody_sync(ctx)
    ftol, gtol = (1e-4, 1e-4) if prec else (1e-11, 1e-10)
    a_ref, phi_ref = oracle.forces(x, m, G=G, eps=eps)
    assert force_rel_err(a.cpu().numpy(), a_ref).max() <= ftol
    assert_elem_close(phi.cpu().numpy(), phi_ref, ftol, "phi")
    for g, o, what in zip(got, oracle.adjoint(x, v, m, G, eps, dt, 1, lx, lv), ("g_x0", "g_v0", "g_m")):
        assert elem_rel_err(g.cpu().numpy(), o, guard=GUARD).max() <= gtol, what


@pytest.mark.parametrize("systems,gradient", [(128, False), (64, True)])
def test_many_large_systems_are_accepted(nb, systems, gradient):
    """Layouts some of whose lists need more than the cap of 4 GiB (systems of 16 384 bodies)."""
    k, G, eps, dt = 16384, 1.1, 0.05, 1e-3
    x1, v1, m1 = inputs.plummer(k, seed=5)
    scale = 1.0 + 0.01 * np.arange(systems)[:, None, None]
    x, v = ((scale * t[None]).reshape(-1, 3) for t in (x1, v1))
    m = np.tile(m1, systems)
    ctx = nb.nbody_init(G=G, eps=eps, dt=dt, offsets=[k * s for s in range(systems + 1)])
    xt, vt, mt = to_dev(x, v, m)
    a, _ = nb.nbody_forces(ctx, xt, mt, with_phi=False)
    nb.nbody_sync(ctx)
    idx = inputs.sample_indices(k, 128, seed=1)
    for s in (0, systems // 2, systems - 1):
        sl = slice(k * s, k * (s + 1))
        a_ref, _ = oracle.forces_at(x[sl], m[sl], idx, G=G, eps=eps)
        assert force_rel_err(a[sl].cpu().numpy()[idx], a_ref).max() <= 1e-4
    if gradient:
        rng = np.random.default_rng(1)
        lx, lv = rng.standard_normal(x.shape), 0.1 * rng.standard_normal(x.shape)
        got = nb.nbody_adjoint(ctx, xt, vt, mt, 1, 1, *to_dev(lx, lv))
        nb.nbody_sync(ctx)
        sl = slice(k * (systems - 1), k * systems)
        for g, o, what in zip(got, oracle.adjoint(x[sl], v[sl], m[sl], G, eps, dt, 1, lx[sl], lv[sl]), ("x", "v", "m")):
            assert elem_rel_err(g[sl].cpu().numpy(), o, guard=GUARD).max() <= 1e-4, what


@pytest.mark.parametrize("capture", ["context", "caller"])
def test_sym64_replays_do_not_depend_on_earlier_masses(nb, tmp_path, monkeypatch, capture):
    """A replay with equal masses right after one with unequal masses gives the bits of an eager call."""
    import torch
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    n, systems, dt = 500, 3, 1e-3
    ens = inputs.ensemble(systems, seed=8, sizes=np.full(systems, n))
    kw = dict(G=1.1, eps=0.05, dt=dt, offsets=[int(o) for o in ens.offsets], precision=nb.FP64)
    eager = nb.nbody_init(**kw)
    assert nb.nbody_get_slicing(eager)["tail"] >= 2
    replayed = nb.nbody_init(flags=nb.FLAG_GRAPH if capture == "context" else 0, **kw)
    unequal = _masses(ens.m, "lognormal", 8)
    first_unequal = ens.m.copy()
    first_unequal[:n] = unequal[:n]

    def buffers():
        xt, vt, mt = to_dev(ens.x, ens.v, ens.m)
        return xt, vt, mt, torch.empty_like(xt)

    def load(b, masses):
        for t, src in zip(b, (ens.x, ens.v, masses)):
            t.copy_(torch.from_numpy(src))

    def step(ctx, b):
        nb.nbody_step(ctx, *b, False, 2)

    r, e = buffers(), buffers()
    graph = torch.cuda.CUDAGraph()
    if capture == "caller":
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            step(replayed, r)
        side.synchronize()
        with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
            step(replayed, r)
    for masses in (unequal, ens.m, first_unequal, ens.m, unequal, first_unequal):
        load(r, masses), load(e, masses)
        torch.cuda.synchronize()
        graph.replay() if capture == "caller" else step(replayed, r)
        step(eager, e)
        torch.cuda.synchronize()
        for got, want in zip(r, e):
            assert torch.equal(got, want)


@pytest.mark.parametrize("sizes", [[0, 130, 1, 300, 64, 1100, 0, 513, 2, 129, 128], [127, 300] * 120, [64] * 300],
                         ids=["uneven", "240", "64x300"])
@pytest.mark.parametrize("tiling", [{}, dict(block=128, i_per_thread=1, j_tile=128, slice=32, variant=2)],
                         ids=["tuned", "many-slots"])
def test_many_small_systems(nb, tiling, sizes):
    """Every system's origin and scales, forces, energies, virials and gradients, with few slots per body (wide
    chunks, two threads a body above 32 768 of them) and with many; a second call gives the same bits."""
    import torch
    G, eps, dt = 1.1, 0.05, 1e-3
    ens = inputs.ensemble(len(sizes), seed=4, sizes=np.array(sizes))
    off = [int(o) for o in ens.offsets]
    x, v, m = ens.x + 30.0 * np.repeat(np.arange(len(sizes)), sizes)[:, None], ens.v, ens.m.copy()
    m[off[1]:off[2]] *= np.exp(np.random.default_rng(1).standard_normal(sizes[1]))
    rng = np.random.default_rng(2)
    lx, lv = rng.standard_normal(x.shape), 0.1 * rng.standard_normal(x.shape)
    ctx = nb.nbody_init(G=G, eps=eps, dt=dt, offsets=off, **tiling)
    xt, vt, mt, lxt, lvt = to_dev(x, v, m, lx, lv)

    def results():
        a, phi = nb.nbody_forces(ctx, xt, mt)
        out = [a, phi, nb.nbody_energy(ctx, xt, vt, mt), nb.nbody_virial(ctx, xt, vt, mt)]
        return out + list(nb.nbody_adjoint_params(ctx, xt, vt, mt, 1, 1, lxt, lvt))

    first, second = results(), results()
    nb.nbody_sync(ctx)
    assert all(torch.equal(s, t) for s, t in zip(first, second))
    a, phi, en, vir, gx, gv, gm, gp = (t.cpu().numpy() for t in first)
    for s in list(range(11)) + [len(sizes) - 1]:
        k = slice(off[s], off[s + 1])
        if sizes[s] < 2:
            assert not a[k].any()
            continue
        a_ref, phi_ref = oracle.forces(x[k], m[k], G=G, eps=eps)
        assert force_rel_err(a[k], a_ref).max() <= 1e-4, s
        assert_elem_close(phi[k], phi_ref, 3e-5, f"phi {s}")
        np.testing.assert_allclose(en[s, 1:3], oracle.energy(x[k], v[k], m[k], G=G, eps=eps)[1:3], rtol=1e-6)
        ox, ov, om, (oG, oe) = oracle.adjoint_params(x[k], v[k], m[k], G, eps, dt, 1, lx[k], lv[k])
        for g, o, what in ((gx, ox, "g_x0"), (gv, ov, "g_v0"), (gm, om, "g_m")):
            assert elem_rel_err(g[k], o, guard=GUARD).max() <= 1e-4, f"{what} {s}"
        scale = max(abs(oG), abs(oe) * eps)
        assert abs(gp[s, 0] - oG) <= 1e-4 * scale and abs(gp[s, 1] - oe) * eps <= 1e-4 * scale, s


def test_sym64_pair_force_to_a_few_ulp(nb, tmp_path, monkeypatch):
    """Two-body systems at separations over eight decades against 50-digit arithmetic. With u = 2^-53: s^2 has three
    roundings, 4.5 u in s^-3, whose own steps are good to 1.5 ulp = 3 u; two products one each: 9.5 u in all,
    and for the potential 6.5 u."""
    from decimal import Decimal, getcontext
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    getcontext().prec = 50
    systems = 500
    rng = np.random.default_rng(3)
    d = rng.standard_normal((systems, 3)) * 10.0 ** rng.uniform(-4, 4, (systems, 1))
    x = np.zeros((2 * systems, 3))
    x[1::2] = d
    m = rng.uniform(0.5, 2.0, 2 * systems)
    # (a third system size keeps the typical size above that of the symmetric pass)
    big, _, big_m = inputs.plummer(200, seed=1)
    off = list(range(0, 2 * systems + 1, 2)) + [2 * systems + 200]
    ctx = _forced(nb, tmp_path / "tune", {"force": (64, 1, 64, 32, 3, 0)}, G=1.0, eps=0.0, dt=1e-3, offsets=off,
                  precision=nb.FP64)
    assert nb.nbody_get_slicing(ctx)["tail"] >= 2
    a, phi = nb.nbody_forces(ctx, *to_dev(np.concatenate([x, big]), np.concatenate([m, _masses(big_m, "lognormal", 1)])))
    nb.nbody_sync(ctx)
    a, phi, u = a.cpu().numpy(), phi.cpu().numpy(), 2.0 ** -53
    for k in range(systems):
        q = [Decimal(float(v)) for v in d[k]]
        r2 = sum(v * v for v in q)
        for i, sign in ((0, 1), (1, -1)):
            mj = Decimal(float(m[2 * k + 1 - i]))
            for c in range(3):
                want = sign * mj * q[c] / (r2 * r2.sqrt())
                assert abs(Decimal(float(a[2 * k + i, c])) - want) <= abs(want) * Decimal(10 * u)
            want = -mj / r2.sqrt()
            assert abs(Decimal(float(phi[2 * k + i])) - want) <= abs(want) * Decimal(7 * u)
