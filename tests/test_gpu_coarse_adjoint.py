"""Gradients from the nodes of an oversampled map against the oracle's analytic
gradient for given maps and against plans without nodes (a radius hint past which
no axis is oversampled): FP32 tiles and, where the last axis keeps its own evenly
spaced points, the line form; the tensor-core contraction; several species,
occupancies, off-centre crystals, single-point axes, the VJP, and a crystal past
the plan's radius (left to the direct kernels bit for bit).  Tolerances (L2): FP32
1e-5 (sums of some 1e-6 and interpolation at 5e-8 per axis, on weights whose
terms partly cancel), tensor cores 1e-4, ten times the contraction's own error."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A
TOL = {"generic": 1e-5, "separable": 1e-4}
FAR = 1e5


def _t(v):
    return torch.tensor(v, device="cuda:0")


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _axes(shape, steps):
    return [W.linspace_axis(c, n, step=s) if n > 1 else np.array([c]) for c, n, s in zip((0.0, 0.0, 4.0), shape, steps)]


def _grown(plan, call):
    before = plan.info()["workspace_bytes"]
    out = call()
    return out, plan.info()["workspace_bytes"] - before


@pytest.mark.parametrize("path, cells, shape, steps, offset, n_sp", [
    ("generic", 9.0, (80, 63, 48), (0.001, 0.001, 0.001), (0, 0, 0), 1),
    ("generic", 9.0, (65, 130, 9), (0.001, 0.001, 0.02), (17.3, -8.0, 40.4), 3),   # line form
    ("generic", 9.0, (1, 290, 280), (0.0, 0.0005, 0.0005), (0.4, 0.3, -0.4), 2),
    ("separable", 16.0, (400, 45, 46), (0.0005, 0.002, 0.002), (3.3, 0.2, 9.9), 2),
])
def test_gradient(path, cells, shape, steps, offset, n_sp):
    c = W.fcc_sphere(radius_cells=cells, seed=401)
    rng = np.random.default_rng(402)
    xyz = c.xyz + np.array(offset, dtype=np.float64)
    coef = np.concatenate([c.coef, c.coef[:1] * 0.8, c.coef[:1] * 1.3])[:n_sp]
    sp = rng.integers(0, n_sp, len(xyz)).astype(np.int32)
    occ = rng.uniform(0.5, 1.0, len(xyz)).astype(np.float32)
    axes = _axes(shape, steps)
    kw = dict(axes=axes, atom_species=sp, path=path)
    plan, bare = api.Plan(coef, A_LAT, len(xyz), **kw), api.Plan(coef, A_LAT, len(xyz), radius_hint=FAR, **kw)
    x, w = _t(xyz), _t(occ)
    A = bare.amplitude(x, w)
    A = A * _t(np.exp(0.3j * rng.normal(size=len(A))).astype(np.complex64))
    I_obs = (A.abs() ** 2 * _t(rng.uniform(0.6, 1.3, len(A)).astype(np.float32)))
    (loss, g), more = _grown(plan, lambda: plan.backward(x, A, I_obs, w))
    (loss_b, g_b), less = _grown(bare, lambda: bare.backward(x, A, I_obs, w))
    plan.check()
    assert more > less  # the nodes' tables too
    assert loss.item() == loss_b.item()
    assert _rel(g.cpu().numpy(), g_b.cpu().numpy()) < TOL[path]
    sel = rng.choice(len(xyz), 40, replace=False)
    _, ref = oracle.loss_grad_atoms(xyz, W.grid_points(axes), A.cpu().numpy(), I_obs.cpu().numpy(), coef, A_LAT, sel,
                                    species=sp, occ=occ)
    assert _rel(g.cpu().numpy()[sel], ref) < TOL[path]
    G = _t((rng.normal(size=len(A)) + 1j * rng.normal(size=len(A))).astype(np.complex64))
    assert _rel(plan.vjp(x, G, w).cpu().numpy(), bare.vjp(x, G, w).cpu().numpy()) < TOL[path]


@pytest.mark.parametrize("path, shape", [("generic", (80, 60, 50)), ("separable", (400, 45, 46))])
def test_larger_crystal_is_left_to_the_direct_kernels(path, shape):
    c = W.fcc_sphere(radius_cells=16.0 if path == "separable" else 9.0, seed=403)
    axes = _axes(shape, (0.001,) * 3)
    kw = dict(axes=axes, atom_species=c.species, path=path)
    plan, bare = api.Plan(c.coef, A_LAT, len(c.xyz), **kw), api.Plan(c.coef, A_LAT, len(c.xyz), radius_hint=FAR, **kw)
    far = c.xyz.copy()
    far[5] *= 4.0
    A = bare.amplitude(_t(far))
    I_obs = A.abs() ** 2 * 0.9
    for xyz, same in ((far, True), (c.xyz, False), (far, True)):
        g, g_b = plan.backward(_t(xyz), A, I_obs)[1], bare.backward(_t(xyz), A, I_obs)[1]
        assert torch.equal(g, g_b) == same
        assert _rel(g.cpu().numpy(), g_b.cpu().numpy()) < TOL[path]
    plan.check()
