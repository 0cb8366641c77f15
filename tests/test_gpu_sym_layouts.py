"""The symmetric passes over layouts of many bodies: 128-body chunks with 64-body i-tiles."""

import numpy as np
import pytest

import oracle
from paper_2511_02655_gb300 import inputs
from helpers import assert_elem_close, force_rel_err, to_dev
from test_gpu_sym import _masses

pytestmark = pytest.mark.gpu


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
