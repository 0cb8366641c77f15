"""Ranges of the mixed path's float32 staging: systems far from the coordinates' origin or with distant
escapers, close pairs in them, and large weights in a gradient."""

import numpy as np
import pytest

import oracle
from paper_2511_02655_gb300 import inputs
from helpers import assert_elem_close, force_rel_err, to_dev
from test_gpu_sym import _forced

pytestmark = pytest.mark.gpu

TOL = 1e-4  # per element, as test_gpu_adjoint.py


def _tight_pairs(npair, eps, seed):
    """A Plummer sphere each of whose bodies has a partner at about half the softening length."""
    x, v, m = inputs.plummer(npair, seed=seed)
    rng = np.random.default_rng(seed)
    x = np.concatenate([x, x + 0.5 * eps * rng.standard_normal(x.shape)])
    return x, np.concatenate([v, v]), np.concatenate([m, m]) * np.exp(0.3 * rng.standard_normal(2 * npair)) / 2


SYM = "symmetric"  # the kernels of the symmetric pass, whatever the size; otherwise nbody_init's variant


def _context(nb, variant, path, monkeypatch, use, **kw):
    if variant != SYM:
        return nb.nbody_init(variant=variant, **kw)
    monkeypatch.setenv("NBODY_TUNE_CACHE", str(path))
    return _forced(nb, path, {"force": (128, 2, 256, 64, 3, 1), "vjp": (128, 2, 128, 64, 3, 1)}, use=use, **kw)


def _check_gradient(nb, x, v, m, G, eps, dt, lx, lv, variant, path, monkeypatch, at=slice(None)):
    args = to_dev(x, v, m) + (1, 1) + to_dev(lx, lv)
    ctx = _context(nb, variant, path, monkeypatch, lambda c: nb.nbody_adjoint(c, *args), G=G, eps=eps, dt=dt, n=len(m))
    got = nb.nbody_adjoint_params(ctx, *args)
    nb.nbody_sync(ctx)
    ctx.close()
    ox, ov, om, (oG, oe) = oracle.adjoint_params(x, v, m, G, eps, dt, 1, lx, lv)
    for g, o, what in zip(got, (ox, ov, om), ("g_x0", "g_v0", "g_m")):
        assert_elem_close(g.cpu().numpy()[at], o[at], TOL, what)
    gG, ge = got[3].cpu().numpy()[0]
    scale = max(abs(oG), abs(oe) * eps)
    assert abs(gG - oG) <= TOL * scale and abs(ge - oe) * eps <= TOL * scale


@pytest.mark.parametrize("variant", [SYM, 0, 1, 2])
@pytest.mark.parametrize("offset", [1e6, 1e8])
def test_gradient_far_from_the_origin(nb, tmp_path, monkeypatch, variant, offset):
    """The staging scale follows the system's extent about its own origin, not its place."""
    eps = 1e-3
    x, v, m = _tight_pairs(150, eps, seed=3)
    x = x + offset * np.array([1.0, -0.5, 0.25])
    rng = np.random.default_rng(4)
    lx, lv = rng.standard_normal(x.shape), rng.standard_normal(x.shape)
    _check_gradient(nb, x, v, m, 1.0, eps, 1e-4, lx, lv, variant, tmp_path / "tune", monkeypatch)


@pytest.mark.parametrize("variant", [SYM, 0, 2])
@pytest.mark.parametrize("far,eps", [(1e9, 1e-3), (1e13, 1e-3), (1e18, 1e-3), (1e10, 1e-5)])
def test_core_beside_a_distant_test_body(nb, tmp_path, monkeypatch, variant, far, eps):
    """One massless body far out: the core's forces and gradients stay what they are."""
    x, v, m = _tight_pairs(150, eps, seed=5)
    x[-1], m[-1] = (far, -far, 0.5 * far), 0.0
    rng = np.random.default_rng(6)
    lx, lv = rng.standard_normal(x.shape), rng.standard_normal(x.shape)
    core = slice(0, len(m) - 1)
    ctx = _context(nb, variant, tmp_path / "tune", monkeypatch, None, G=1.0, eps=eps, dt=1e-4, n=len(m))
    a, _ = nb.nbody_forces(ctx, *to_dev(x, m))
    nb.nbody_sync(ctx)
    ctx.close()
    a_ref, _ = oracle.forces(x, m, G=1.0, eps=eps)
    assert force_rel_err(a.cpu().numpy()[core], a_ref[core]).max() <= 1e-4
    if variant == 0:
        b, _ = nb.nbody_forces_noalloc(*to_dev(x, m), 1.0, eps)
        assert force_rel_err(b.cpu().numpy()[core], a_ref[core]).max() <= 1e-4
    _check_gradient(nb, x, v, m, 1.0, eps, 1e-4 if eps == 1e-3 else 1e-9, lx, lv, variant,
                    tmp_path / "tune", monkeypatch, core)


@pytest.mark.parametrize("variant", [SYM, 0, 2])
@pytest.mark.parametrize("n", [65, 300])
def test_large_weights(nb, tmp_path, monkeypatch, variant, n):
    """Weights of 1e19 beside the padding of partial tiles."""
    x, v, m = inputs.plummer(n, seed=7)
    rng = np.random.default_rng(8)
    lx, lv = 1e19 * rng.standard_normal((n, 3)), 1e19 * rng.standard_normal((n, 3))
    _check_gradient(nb, x, v, m, 1.1, 0.05, 1e-2, lx, lv, variant, tmp_path / "tune", monkeypatch)
