"""Adjoint over the clusters of an S list against the oracle's analytic gradient
for given maps and against the direct kernel of a plan without clusters: one and
three species, occupancies, off-centre crystals, point counts around the 64- and
256-point tiles of a cluster, a volume of points, a line, a factor table, a
crystal past the plan's radius, and the VJP.  Tolerance 2e-5 (L2): MUFU sin/cos
(2^-21 absolute) per (atom, cluster), neglected columns of 2e-6 at the ball's
surface, FP32 polynomials of some 1e-6, summed over tens of clusters."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A
TOL = 2e-5


def _t(v):
    return torch.tensor(v, device="cuda:0")


def _rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _check(xyz, sp, coef, S, occ=None, radius_hint=0.0, clustered=True):
    rng = np.random.default_rng(len(S))
    A = (oracle.amplitude(xyz, S, coef, A_LAT, species=sp, occ=occ) * np.exp(0.3j * rng.normal(size=len(S)))).astype(np.complex64)
    I_obs = (np.abs(A) ** 2 * rng.uniform(0.6, 1.3, len(S))).astype(np.float32)
    kw = dict(s_list=S, atom_species=sp)
    plan = api.Plan(coef, A_LAT, len(xyz), radius_hint=radius_hint, **kw)
    bare = api.Plan(coef, A_LAT, len(xyz), split_k=1, **kw)
    x, w = _t(xyz), None if occ is None else _t(occ)
    loss, g = plan.backward(x, _t(A), _t(I_obs), w)
    loss_b, g_b = bare.backward(x, _t(A), _t(I_obs), w)
    plan.check()
    bare.check()
    assert loss.item() == loss_b.item()
    sel = rng.choice(len(xyz), min(150, len(xyz)), replace=False)
    _, ref = oracle.loss_grad_atoms(xyz, S, A, I_obs, coef, A_LAT, sel, species=sp, occ=occ)
    g, g_b = g.cpu().numpy(), g_b.cpu().numpy()
    assert _rel(g[sel], ref) < TOL
    assert _rel(g, g_b) < TOL
    G = _t((rng.normal(size=len(S)) + 1j * rng.normal(size=len(S))).astype(np.complex64))
    v, v_b = plan.vjp(x, G, w).cpu().numpy(), bare.vjp(x, G, w).cpu().numpy()
    assert _rel(v, v_b) < TOL
    assert np.array_equal(v, v_b) != clustered


@pytest.mark.parametrize("points, radius, offset, n_sp", [
    (20000, 9.5, (0, 0, 0), 1), (30011, 9.0, (17.3, -8.0, 40.4), 3), (16385, 11.3, (0.4, 0.3, -0.4), 2),
])
def test_detector_patch(points, radius, offset, n_sp):
    c = W.fcc_sphere(radius_cells=radius, seed=191)
    xyz = c.xyz + np.array(offset, dtype=np.float64)
    rng = np.random.default_rng(192)
    coef = np.concatenate([c.coef, c.coef[:1] * 0.8, c.coef[:1] * 1.3])[:n_sp]
    sp = rng.integers(0, n_sp, len(xyz)).astype(np.int32)
    occ = rng.uniform(0.5, 1.0, len(xyz)).astype(np.float32)
    _check(xyz, sp, coef, W.ewald_slice(points, rocking_deg=0.02, seed=193), occ)


def test_volume_and_line():
    c = W.fcc_sphere(radius_cells=9.0, seed=194)
    rng = np.random.default_rng(195)
    _check(c.xyz, c.species, c.coef, np.array([1.0, 1.0, 1.0]) + rng.uniform(-0.02, 0.02, (20000, 3)))
    _check(c.xyz, c.species, c.coef,
           np.array([2.0, 0.0, 0.0]) + rng.uniform(-0.2, 0.2, (20000, 1)) * np.array([[0.3, -0.7, 0.2]]))


def test_larger_crystal_is_left_to_the_direct_kernel():
    c = W.fcc_sphere(radius_cells=9.0, seed=196)
    _check(c.xyz, c.species, c.coef, W.ewald_slice(20000, seed=197), radius_hint=4.0, clustered=False)


def test_factor_table():
    m = W.fcc_cell_blocks(n=(12, 12, 12))
    S = W.ewald_slice(20000, seed=198)
    rng = np.random.default_rng(199)
    T = rng.normal(size=(2, len(S))) + 1j * rng.normal(size=(2, len(S)))
    plan = api.Plan(W.si_ge_species(), A_LAT, len(m.origins), s_list=S, atom_species=m.types, factor_table=T)
    I_obs = (np.abs(oracle.amplitude_table(m.origins, S, T, types=m.types)) ** 2 * rng.uniform(0.5, 1.5, len(S))).astype(np.float32)
    x = _t(m.origins)
    _, g = plan.backward(x, plan.amplitude(x), _t(I_obs))
    assert _rel(g.cpu().numpy(), oracle.loss_grad_table(m.origins, S, I_obs, T, types=m.types)[1]) < 1e-3
