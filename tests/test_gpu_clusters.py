"""Clustered S lists against the oracle: detector patches of one and of several
clusters, two species, occupancies, off-centre crystals, volumes of points, a
factor table, uneven batches of clustered and direct instances, and crystals
past the plan's radius (left to the direct kernels).  Tolerance 1e-5: MUFU
sin/cos (2^-21 absolute per term), FP32 sums over at most 512 atoms and
neglected terms of 2e-6 at the ball's surface, ten times inside the FP32
paths' 1e-4."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A
TOL = 1e-5


def _t(v):
    return torch.tensor(v, device="cuda:0")


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))



def _check(c, xyz, S, occ=None, radius_hint=0.0, n=500):
    plan = api.Plan(c.coef, A_LAT, len(xyz), s_list=S, atom_species=c.species, radius_hint=radius_hint)
    bare = api.Plan(c.coef, A_LAT, len(xyz), s_list=S, atom_species=c.species, split_k=1)
    args = (_t(xyz), None if occ is None else _t(occ))
    A, I = plan.amplitude(*args).cpu().numpy(), plan.intensity(*args).cpu().numpy()
    plan.check()
    idx = np.random.default_rng(1).choice(len(S), min(n, len(S)), replace=False)
    ref = oracle.amplitude(xyz, S[idx], c.coef, A_LAT, species=c.species, occ=occ)
    assert _rel(A[idx], ref) < TOL
    assert _rel(I[idx], np.abs(ref) ** 2) < 2 * TOL
    assert _rel(A, bare.amplitude(*args).cpu().numpy()) < TOL  # every point, against the direct kernels
    return plan, bare


@pytest.mark.parametrize("points, radius, offset", [
    (20000, 9.5, (0, 0, 0)), (60001, 9.0, (17.3, -8.0, 40.4)), (30011, 12.3, (0.4, 0.3, -0.4)), (100003, 6.0, (0, 0, 0)),
])
def test_detector_patch(points, radius, offset):
    c = W.fcc_sphere(radius_cells=radius, seed=91)
    xyz = c.xyz + np.array(offset, dtype=np.float64)
    occ = np.random.default_rng(92).uniform(0.5, 1.0, len(xyz)).astype(np.float32)
    plan, bare = _check(c, xyz, W.ewald_slice(points, rocking_deg=0.02, seed=93), occ)
    assert plan.info()["workspace_bytes"] > bare.info()["workspace_bytes"] + 1000000  # its clusters


def test_volume_of_points_and_a_line():
    c = W.fcc_sphere(radius_cells=9.0, seed=94)
    rng = np.random.default_rng(95)
    _check(c, c.xyz, np.array([1.0, 1.0, 1.0]) + rng.uniform(-0.02, 0.02, (40000, 3)))
    _check(c, c.xyz, np.array([2.0, 0.0, 0.0]) + rng.uniform(-0.2, 0.2, (50000, 1)) * np.array([[0.3, -0.7, 0.2]]))
    _check(c, c.xyz, np.tile([[1.01, 1.0, 0.98]], (40000, 1)))  # one cluster without extent


def test_larger_crystal_is_left_to_the_direct_kernels():
    c = W.fcc_sphere(radius_cells=9.0, seed=96)
    S = W.ewald_slice(30000, seed=97)
    far = c.xyz.copy()
    far[5] *= 4.0  # one atom far past the compact crystal's radius
    far[77] *= -3.5
    _check(c, far, S)
    _check(c, c.xyz, S, radius_hint=4.0)  # a hint that the crystal breaks


def test_factor_table():
    m = W.fcc_cell_blocks(n=(12, 12, 12))
    S = W.ewald_slice(40000, seed=98)
    rng = np.random.default_rng(99)
    T = rng.normal(size=(2, len(S))) + 1j * rng.normal(size=(2, len(S)))
    plan = api.Plan(W.si_ge_species(), A_LAT, len(m.origins), s_list=S, atom_species=m.types, factor_table=T)
    A = plan.amplitude(_t(m.origins)).cpu().numpy()
    idx = rng.choice(len(S), 600, replace=False)
    assert _rel(A[idx], oracle.amplitude_table(m.origins, S[idx], T[:, idx], types=m.types)) < TOL


def test_uneven_batch():
    xyz, sp, coef, S, ao, so = W.ewald_batch(7, (300, 20000), (150, 60000), seed=3100)
    xyz[ao[3]] *= 9.0  # instance 3 grows past its radius
    plan = api.Plan(coef, A_LAT, len(xyz), s_list=S, atom_species=sp, atom_off=ao, s_off=so)
    A = plan.amplitude(_t(xyz)).cpu().numpy()
    for _ in range(2):
        again = plan.amplitude(_t(xyz)).cpu().numpy()
    plan.check()
    assert np.array_equal(A.view(np.float32), again.view(np.float32))
    for b in range(7):
        idx = so[b] + np.random.default_rng(b).choice(so[b + 1] - so[b], min(300, so[b + 1] - so[b]), replace=False)
        ref = oracle.amplitude(xyz[ao[b]:ao[b + 1]], S[idx], coef, A_LAT, species=sp[ao[b]:ao[b + 1]])
        assert _rel(A[idx], ref) < TOL, b
