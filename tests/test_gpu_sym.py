"""The symmetric all-pairs passes (every unordered pair once) at the edges of their tiles.

They are chosen by the tuner only, so the tiling under test is put into the tuning cache
(NBODY_TUNE_CACHE) under the key that a first context of the same setup writes."""

import numpy as np
import pytest

import oracle
from paper_2511_02655_gb300 import inputs
from helpers import assert_elem_close, force_rel_err, to_dev

pytestmark = pytest.mark.gpu

MIX_MED, MIX_MAX, MIX_PHI_MAX = 1e-6, 1e-4, 3e-5  # the mixed path's bounds (test_gpu_parity.py)


def _forced(nb, path, tilings, use=None, **kw):
    """A context whose tilings ({"force" | "vjp": cache line}) come from the tuning cache."""
    if path.exists():
        path.unlink()
    ctx = nb.nbody_init(**kw)
    if use:
        use(ctx)  # first use of a kernel that is tuned late
    ctx.close()
    lines = []
    for line in path.read_text().splitlines():
        key = line.split("\t")[0]
        for kind, t in tilings.items():
            if f"|{kind}|" in key:
                lines.append(key + "\t" + " ".join(str(v) for v in t))
    path.write_text("\n".join(lines) + "\n")
    return nb.nbody_init(**kw)


def _masses(m, kind, seed):
    return m if kind == "equal" else m * np.exp(0.4 * np.random.default_rng(seed).standard_normal(len(m)))


# block, i-bodies per lane, j-tile, slice, variant, tail: i-tiles of 256, 512, 512 and 1024 bodies
TILINGS = [(128, 2, 256, 64, 3, 0), (128, 4, 256, 192, 3, 1), (256, 2, 256, 320, 3, 2), (256, 4, 256, 64, 3, 1)]


@pytest.mark.parametrize("tiling", TILINGS)
@pytest.mark.parametrize("n", [1, 2, 63, 65, 257, 1025, 4999])
@pytest.mark.parametrize("masses", ["equal", "lognormal"])
def test_sym_forces(nb, tmp_path, monkeypatch, tiling, n, masses):
    import torch
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    G, eps = 1.2, 0.05  # 4 eps = 0.2: near pairs in most tiles
    x, v, m = inputs.plummer(n, seed=n)
    m = _masses(m, masses, n)
    ctx = _forced(nb, tmp_path / "tune", {"force": tiling}, G=G, eps=eps, dt=1e-3, n=n)
    assert nb.nbody_get_slicing(ctx)["tail"] >= 2
    xt, mt = to_dev(x, m)
    a, phi = nb.nbody_forces(ctx, xt, mt)
    a0, _ = nb.nbody_forces(ctx, xt, mt, with_phi=False)
    nb.nbody_sync(ctx)
    assert torch.equal(a, a0)
    if n == 1:
        assert not a.any() and not phi.any()
        return
    a_ref, phi_ref = oracle.forces(x, m, G=G, eps=eps)
    e = force_rel_err(a.cpu().numpy(), a_ref)
    assert np.median(e) <= MIX_MED and e.max() <= MIX_MAX, (np.median(e), e.max())
    assert_elem_close(phi.cpu().numpy(), phi_ref, MIX_PHI_MAX, "phi")


@pytest.mark.parametrize("tiling", TILINGS)
def test_sym_lennard_jones(nb, tmp_path, monkeypatch, tiling):
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    x, v, m, box = inputs.lj_gas(2050, seed=7, density=0.3)
    m = _masses(m, "lognormal", 3)
    ctx = _forced(nb, tmp_path / "tune", {"force": tiling}, law=nb.LENNARD_JONES, dt=1e-3, n=2050, lj_epsilon=1.3,
                  lj_sigma=0.9)
    assert nb.nbody_get_slicing(ctx)["tail"] >= 2
    a, phi = nb.nbody_forces(ctx, *to_dev(x, m))
    nb.nbody_sync(ctx)
    a_ref, phi_ref = oracle.lj_forces(x, m, eps_lj=1.3, sigma=0.9)
    e = force_rel_err(a.cpu().numpy(), a_ref)
    assert np.median(e) <= MIX_MED and e.max() <= MIX_MAX, (np.median(e), e.max())
    assert_elem_close(phi.cpu().numpy(), phi_ref, MIX_MAX, "phi")


# i-tiles of 64, 128, 256 and 256 bodies
TILINGS64 = [(64, 1, 64, 32, 3, 0), (128, 1, 64, 96, 3, 1), (256, 1, 64, 64, 3, 0), (128, 2, 64, 160, 3, 1)]


@pytest.mark.parametrize("tiling", TILINGS64)
@pytest.mark.parametrize("n", [65, 300, 1025, 2500])
@pytest.mark.parametrize("length,mass", [(1.0, 1.0), (1e100, 1e30), (1e-95, 1.0)])
@pytest.mark.parametrize("masses", ["equal", "lognormal"])
def test_sym64_forces(nb, tmp_path, monkeypatch, tiling, n, length, mass, masses):
    """FP64 path, in units where s^2 takes the integer steps and in some where it leaves their
    range (the oracle gets scaled copies; powers of ten, so the comparison is good to rounding)."""
    import torch
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    x, v, m = inputs.plummer(n, seed=n)
    m = _masses(m, masses, n)
    xs, ms, eps = x * length, m * mass, 0.03 * length
    ctx = _forced(nb, tmp_path / "tune", {"force": tiling}, G=1.1, eps=eps, dt=1e-3, n=n, precision=nb.FP64)
    assert nb.nbody_get_slicing(ctx)["tail"] >= 2
    xt, mt = to_dev(xs, ms)
    a, phi = nb.nbody_forces(ctx, xt, mt)
    a0, _ = nb.nbody_forces(ctx, xt, mt, with_phi=False)
    nb.nbody_sync(ctx)
    assert torch.equal(a, a0)
    a_ref, phi_ref = oracle.forces(x, m, G=1.1, eps=0.03)
    a, phi = a.cpu().numpy() * (length / mass) * length, phi.cpu().numpy() * (length / mass)
    assert force_rel_err(a, a_ref).max() <= 1e-12
    assert_elem_close(phi, phi_ref, 1e-12, "phi")


@pytest.mark.parametrize("n,split", [(65, 4), (700, 4), (1400, 2), (2050, 1)])
@pytest.mark.parametrize("law", [0, 1])
def test_sym64_shared_blocks(nb, tmp_path, monkeypatch, law, n, split):
    """Lists short enough that 4, 2 or 1 warps share a block's rotation: forces, potentials and gradients."""
    import torch
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    rows = -(-n // 64)
    items = sum((n - 64 * r + 31) // 32 for r in range(rows))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert split == (4 if 8 * items <= 16 * sms else 2 if 4 * items <= 16 * sms else 1)
    x, v, m = inputs.lj_gas(n, seed=3)[:3] if law else inputs.plummer(n, seed=n)
    m = _masses(m, "lognormal", n)
    kw = dict(law=1, dt=1e-3, n=n, lj_epsilon=1.3, lj_sigma=0.9) if law else dict(G=1.1, eps=0.03, dt=1e-3, n=n)
    rng = np.random.default_rng(n)
    lx, lv = rng.standard_normal((n, 3)), 0.1 * rng.standard_normal((n, 3))
    args = to_dev(x, v, m) + (2, 2) + to_dev(lx, lv)
    lines = {"force": (64, 1, 64, 1, 3, 0)}
    if not law:
        lines["vjp"] = (64, 1, 64, 1, 3, 0)
    ctx = _forced(nb, tmp_path / "tune", lines, precision=nb.FP64,
                  **({} if law else {"use": lambda c: nb.nbody_adjoint(c, *args)}), **kw)
    a, phi = nb.nbody_forces(ctx, *to_dev(x, m))
    nb.nbody_sync(ctx)
    assert nb.nbody_get_slicing(ctx)["n_items"] == items
    ref = oracle.lj_forces(x, m, eps_lj=1.3, sigma=0.9) if law else oracle.forces(x, m, G=1.1, eps=0.03)
    tol = 1e-10 if law else 1e-12
    assert force_rel_err(a.cpu().numpy(), ref[0]).max() <= tol
    assert_elem_close(phi.cpu().numpy(), ref[1], tol, "phi")
    if not law:
        gx, gv, gm = nb.nbody_adjoint(ctx, *args)
        nb.nbody_sync(ctx)
        for got, want, name in zip((gx, gv, gm), oracle.adjoint(x, v, m, 1.1, 0.03, 1e-3, 2, lx, lv), ("x", "v", "m")):
            assert_elem_close(got.cpu().numpy(), want, 1e-11, name)


def test_sym64_masses_change_between_calls(nb):
    """Equal masses are recognised anew in every call, replayed graphs included."""
    import torch
    n, G, eps, dt = 700, 1.0, 0.05, 1e-3
    x, v, m = inputs.plummer(n, seed=8)
    m2 = _masses(m, "lognormal", 8)
    ctx = nb.nbody_init(G=G, eps=eps, dt=dt, n=n, precision=nb.FP64, energy_every=2, flags=nb.FLAG_GRAPH)
    assert nb.nbody_get_slicing(ctx)["tail"] >= 2
    xt, vt, mt = to_dev(x, v, m)
    at = torch.empty_like(xt)
    log = torch.empty((1, 1, 9), dtype=torch.float64, device="cuda")
    for masses in (m, m2, m, m2, m2):
        for t, src in ((xt, x), (vt, v), (mt, masses)):
            t.copy_(torch.from_numpy(src))
        nb.nbody_step(ctx, xt, vt, mt, at, False, 2, log)
        a, _ = nb.nbody_forces(ctx, xt, mt)
        nb.nbody_sync(ctx)
        xr, vr, ar, lr = oracle.kdk(x, v, masses, G, eps, dt, 2, energy_every=2)
        assert np.abs(xt.cpu().numpy() - xr).max() <= 1e-13
        assert force_rel_err(at.cpu().numpy(), ar).max() <= 1e-12
        assert force_rel_err(a.cpu().numpy(), ar).max() <= 1e-12
        np.testing.assert_allclose(log.cpu().numpy()[0, 0, 0:3], lr[0, 0:3], rtol=1e-12)


@pytest.mark.parametrize("tiling", TILINGS64)
def test_sym64_lennard_jones_and_coincident(nb, tmp_path, monkeypatch, tiling):
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    x, v, m, box = inputs.lj_gas(1100, seed=7, density=0.3)
    m = _masses(m, "lognormal", 3)
    kw = dict(law=nb.LENNARD_JONES, dt=1e-3, n=1100, lj_epsilon=1.3, lj_sigma=0.9, precision=nb.FP64)
    ctx = _forced(nb, tmp_path / "tune", {"force": tiling}, **kw)
    assert nb.nbody_get_slicing(ctx)["tail"] >= 2
    a, phi = nb.nbody_forces(ctx, *to_dev(x, m))
    nb.nbody_sync(ctx)
    a_ref, phi_ref = oracle.lj_forces(x, m, eps_lj=1.3, sigma=0.9)
    assert force_rel_err(a.cpu().numpy(), a_ref).max() <= 1e-12
    assert_elem_close(phi.cpu().numpy(), phi_ref, 1e-12, "phi")
    # unsoftened coincident bodies stay a reported condition
    ctx = _forced(nb, tmp_path / "tune", {"force": tiling}, G=1.0, eps=0.0, dt=1e-3, n=1100, precision=nb.FP64)
    x[700] = x[3]
    nb.nbody_forces(ctx, *to_dev(x, m))
    with pytest.raises(nb.NBodyError) as ei:
        nb.nbody_sync(ctx)
    assert ei.value.status == 5


@pytest.mark.parametrize("length,mass", [(1e12, 1e30), (1e-9, 1e-27), (1.0, 1.0)])
def test_mixed_forces_in_any_units(nb, length, mass):
    """Staging scales positions and masses by powers of two, so the float32 arithmetic stays in
    range in any units (metres and kilograms of a planetary system included)."""
    n = 3000
    x, v, m = inputs.plummer(n, seed=5)
    m = _masses(m, "lognormal", 5)
    for variant in (0, 1, 2):
        ctx = nb.nbody_init(G=1.0, eps=0.02 * length, dt=1e-3, n=n, variant=variant)
        a, phi = nb.nbody_forces(ctx, *to_dev(x * length, m * mass))
        nb.nbody_sync(ctx)
        a_ref, phi_ref = oracle.forces(x, m, G=1.0, eps=0.02)
        e = force_rel_err(a.cpu().numpy() * (length / mass * length), a_ref)
        assert np.median(e) <= MIX_MED and e.max() <= MIX_MAX, (variant, np.median(e), e.max())
        assert_elem_close(phi.cpu().numpy() * (length / mass), phi_ref, MIX_PHI_MAX, "phi")
        ctx.close()


@pytest.mark.parametrize("law", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
def test_reported_tiling_can_be_requested(nb, law, prec):
    """Whatever the tuner chose, what nbody_get_tuning reports is a valid request."""
    n = 4500
    x, v, m, box = inputs.lj_gas(n, seed=3) if law else inputs.plummer(n, seed=3) + (0.0,)
    kw = dict(law=law, precision=prec, n=n, dt=1e-3, eps=0.0 if law else 0.02)
    ctx = nb.nbody_init(**kw)
    a, _ = nb.nbody_forces(ctx, *to_dev(x, m))
    assert nb.nbody_get_slicing(ctx)["tail"] >= 2 or prec == 1
    t = nb.nbody_get_tuning(ctx)
    again = nb.nbody_init(block=t["block"], i_per_thread=t["i_per_thread"], j_tile=t["j_tile"], slice=t["slice"],
                          variant=t["variant"], **kw)
    b, _ = nb.nbody_forces(again, *to_dev(x, m))
    nb.nbody_sync(again)
    assert force_rel_err(b.cpu().numpy(), a.cpu().numpy()).max() <= (1e-4 if prec else 1e-12)


def test_sym_several_systems_and_zero_masses(nb, tmp_path, monkeypatch):
    """Systems of every kind in one list: empty, single, equal masses, unequal ones, massless bodies
    (they feel forces and exert none), one far from the origin."""
    import torch
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    sizes = [0, 1, 300, 1100, 2, 700, 0, 513]
    ens = inputs.ensemble(len(sizes), seed=3, sizes=np.array(sizes))
    off = [int(o) for o in ens.offsets]
    x, m = ens.x.copy(), ens.m.copy()
    m[off[3]:off[4]:2] = 0.0
    m[off[5]:off[6]] *= np.exp(np.random.default_rng(1).standard_normal(700))
    x[off[7]:off[8]] += 50.0
    ctx = _forced(nb, tmp_path / "tune", {"force": (128, 2, 256, 128, 3, 1)}, G=1.0, eps=0.02, dt=1e-3, offsets=off)
    assert nb.nbody_get_slicing(ctx)["tail"] >= 2
    xt, mt = to_dev(x, m)
    a, phi = nb.nbody_forces(ctx, xt, mt)
    a2, phi2 = nb.nbody_forces(ctx, xt, mt)
    nb.nbody_sync(ctx)
    assert torch.equal(a, a2) and torch.equal(phi, phi2)
    for s, k in enumerate(sizes):
        b, e = off[s], off[s + 1]
        if k < 2:
            assert not a[b:e].any()
            continue
        a_ref, phi_ref = oracle.forces(x[b:e], m[b:e], G=1.0, eps=0.02)
        assert force_rel_err(a[b:e].cpu().numpy(), a_ref).max() <= MIX_MAX, s
        assert_elem_close(phi[b:e].cpu().numpy(), phi_ref, MIX_PHI_MAX, f"phi {s}")


@pytest.mark.parametrize("prec,tiling", [(1, (128, 1, 128, 64, 3, 0)), (1, (128, 2, 128, 64, 3, 1)),
                                         (1, (256, 2, 128, 192, 3, 0)), (0, (64, 1, 64, 32, 3, 0)),
                                         (0, (128, 1, 64, 96, 3, 1)), (0, (256, 1, 64, 64, 3, 0))])
@pytest.mark.parametrize("n", [2, 65, 513, 1100])
def test_sym_vjp(nb, tmp_path, monkeypatch, prec, tiling, n):
    """Gradients through a few steps, G and eps included, near pairs in most tiles (4 eps = 0.2)."""
    import torch
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(tmp_path / "tune"))
    G, eps, dt, T, K = 1.1, 0.05, 4e-3, 3, 2
    x, v, m = inputs.plummer(n, seed=70 + n)
    m = _masses(m, "lognormal", n)
    rng = np.random.default_rng(n)
    lx, lv = rng.standard_normal((n, 3)), 0.1 * rng.standard_normal((n, 3))
    args = to_dev(x, v, m) + (T, K) + to_dev(lx, lv)
    ctx = _forced(nb, tmp_path / "tune", {"vjp": tiling}, use=lambda c: nb.nbody_adjoint(c, *args), G=G, eps=eps, dt=dt,
                  n=n, precision=prec)
    gx, gv, gm, gp = nb.nbody_adjoint_params(ctx, *args)
    hx, hv, hm = nb.nbody_adjoint(ctx, *args)
    nb.nbody_sync(ctx)
    assert torch.equal(gx, hx) and torch.equal(gv, hv) and torch.equal(gm, hm)
    ox, ov, om, (oG, oe) = oracle.adjoint_params(x, v, m, G, eps, dt, T, lx, lv)
    tol = 1e-4 if prec else 1e-11  # the bounds of test_gpu_adjoint.py
    for g, o, what in ((gx, ox, "g_x0"), (gv, ov, "g_v0"), (gm, om, "g_m")):
        assert_elem_close(g.cpu().numpy(), o, tol, what)
    gG, ge = gp.cpu().numpy()[0]
    scale = max(abs(oG), abs(oe) * eps)
    assert abs(gG - oG) <= tol * scale and abs(ge - oe) * eps <= tol * scale


@pytest.mark.parametrize("n", [33, 2048, 2049, 8193, 24000, 24001, 524288, 524289])
@pytest.mark.parametrize("masses", ["equal", "lognormal"])
def test_noalloc_work_splits(nb, n, masses):
    """Both sides of every size at which the allocation-free entry point changes its work split,
    against the oracle on sampled bodies."""
    import torch
    x, v, m = inputs.plummer(n, seed=n)
    m = _masses(m, masses, n)
    xt, mt = to_dev(x, m)
    a, phi = nb.nbody_forces_noalloc(xt, mt, 1.1, 0.01, phi=torch.empty_like(mt))
    a0, _ = nb.nbody_forces_noalloc(xt, mt, 1.1, 0.01)
    torch.cuda.synchronize()
    assert torch.equal(a, a0)
    idx = inputs.sample_indices(n, 512, seed=1)
    a_ref, phi_ref = oracle.forces_at(x, m, idx, G=1.1, eps=0.01)
    e = force_rel_err(a.cpu().numpy()[idx], a_ref)
    assert np.median(e) <= MIX_MED and e.max() <= MIX_MAX, (np.median(e), e.max())
    assert_elem_close(phi.cpu().numpy()[idx], phi_ref, MIX_PHI_MAX, "phi")
