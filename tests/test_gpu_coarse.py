"""Oversampled maps (sum at Chebyshev nodes, interpolated) against the oracle and
against plans without nodes (a radius hint past which no axis is oversampled):
node counts below, at and above the 16-node stages and 64-point tiles, axes that
keep their own points, single-point axes, unsorted and uneven axes, off-centre
crystals, occupancies, host calls, captured replays, and crystals past the plan's
radius (left to the direct sum bit for bit).  Tolerances: FP32 2e-6 (sums of
some 1e-7 to 1e-6, three stages of interpolation at 5e-8 and their FP32 rounding);
tensor-core path 1e-4, its own."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A
TOL = {"generic": 2e-6, "separable": 1e-4}
FAR = 1e5  # radius hint without nodes


def _t(v):
    return torch.tensor(v, device="cuda:0")


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _axes(shape, steps, centre=(0.0, 0.0, 4.0)):
    return [W.linspace_axis(c, n, step=s) if n > 1 else np.array([c]) for c, n, s in zip(centre, shape, steps)]


def _plans(c, axes, path, **kw):
    kw.update(axes=axes, atom_species=c.species, path=path)
    plan = api.Plan(c.coef, A_LAT, len(c.xyz), **kw)
    bare = api.Plan(c.coef, A_LAT, len(c.xyz), **dict(kw, radius_hint=FAR))
    return plan, bare


def _nodes(plan, bare):
    return plan.info()["workspace_bytes"] != bare.info()["workspace_bytes"]


@pytest.mark.parametrize("path, cells, shape, steps, offset", [
    ("generic", 9.0, (65, 63, 64), (0.002, 0.002, 0.002), (0, 0, 0)),
    ("generic", 9.0, (1000, 1, 131), (0.0004, 0.0, 0.001), (17.3, -8.0, 40.4)),
    ("generic", 11.0, (3, 190, 97), (0.05, 0.0015, 0.004), (0.4, 0.3, -0.4)),
    ("generic", 12.0, (290, 33, 9), (0.0004, 0.001, 0.02), (0, 0, 0)),
    ("separable", 14.0, (129, 130, 65), (0.002, 0.002, 0.002), (0, 0, 0)),
    ("separable", 14.0, (900, 1, 900), (0.0003, 0.0, 0.0003), (3.3, 0.2, 9.9)),
    ("separable", 16.0, (40, 301, 66), (0.02, 0.001, 0.003), (0, 0, 0)),
])
def test_map_against_oracle_and_direct(path, cells, shape, steps, offset):
    c = W.fcc_sphere(radius_cells=cells, seed=301)
    xyz = c.xyz + np.array(offset, dtype=np.float64)
    axes = _axes(shape, steps)
    occ = np.random.default_rng(302).uniform(0.5, 1.0, len(xyz)).astype(np.float32)
    plan, bare = _plans(c, axes, path)
    assert _nodes(plan, bare)
    x, w = _t(xyz), _t(occ)
    A = plan.amplitude(x, w).cpu().numpy()
    for _ in range(3):  # eager, captured, replayed
        again = plan.amplitude(x, w).cpu().numpy()
        assert np.array_equal(A.view(np.float32), again.view(np.float32))
    H = plan.amplitude_host(xyz, occ)
    torch.cuda.synchronize()
    assert np.array_equal(A.view(np.float32), H.numpy().reshape(-1).view(np.float32))
    plan.check()
    D = bare.amplitude(x, w).cpu().numpy()
    assert _rel(A, D) < TOL[path]
    assert _rel(plan.intensity(x, w).cpu().numpy(), bare.intensity(x, w).cpu().numpy()) < 2 * TOL[path]
    S = W.grid_points(axes)
    idx = np.random.default_rng(303).choice(len(S), 400, replace=False)
    ref = oracle.amplitude(xyz, S[idx], c.coef, A_LAT, species=c.species, occ=occ)
    # against the map's scale: a sample may miss the peak
    scale = np.sqrt(np.mean(np.abs(D) ** 2))
    assert np.sqrt(np.mean(np.abs(A[idx] - ref) ** 2)) < TOL[path] * max(scale, np.sqrt(np.mean(np.abs(ref) ** 2)))


def test_unsorted_and_uneven_axes():
    c = W.fcc_sphere(radius_cells=10.0, seed=304)
    rng = np.random.default_rng(305)
    axes = [rng.uniform(-0.1, 0.1, 90), np.repeat([0.0, 0.03], 40), np.sort(rng.uniform(3.95, 4.1, 70))[::-1].copy()]
    plan, bare = _plans(c, axes, "generic")
    assert _nodes(plan, bare)
    x = _t(c.xyz)
    assert _rel(plan.amplitude(x).cpu().numpy(), bare.amplitude(x).cpu().numpy()) < TOL["generic"]


@pytest.mark.parametrize("path, shape", [("generic", (80, 60, 50)), ("separable", (140, 140, 65))])
def test_larger_crystal_is_left_to_the_direct_sum(path, shape):
    c = W.fcc_sphere(radius_cells=14.0 if path == "separable" else 9.0, seed=306)
    axes = _axes(shape, (0.002,) * 3)
    plan, bare = _plans(c, axes, path)
    assert _nodes(plan, bare)
    x = c.xyz.copy()
    small = plan.amplitude(_t(x))
    x[5] *= 4.0  # one atom far past the compact crystal's radius
    for p in (plan.amplitude, plan.intensity):
        q = bare.amplitude if p == plan.amplitude else bare.intensity
        assert torch.equal(p(_t(x)), q(_t(x)))
    assert torch.equal(plan.amplitude(_t(c.xyz)), small)  # and back
    plan.check()


@pytest.mark.parametrize("shape, offset", [((150, 150, 24), (0.0, 0.0, 0.0)), ((33, 600, 24), (7.3, -4.6, 3.2))])
def test_grazing_incidence_in_plane(shape, offset):
    c = W.truncated_pyramid(44, 16, 14)
    xyz = c.xyz + np.array(offset)
    gid = dict(wavelength=W.WAVELENGTH_10KEV, alpha_i=W.GID_ALPHA_I, delta=W.GID_DELTA, beta=W.GID_BETA)
    axes = list(W.gid_axes(*shape))
    plan, bare = _plans(c, axes, "separable", gid=gid)
    assert _nodes(plan, bare)
    A, D = plan.amplitude(_t(xyz)).cpu().numpy(), bare.amplitude(_t(xyz)).cpu().numpy()
    assert not np.array_equal(A, D)
    assert _rel(A, D) < 5e-5  # either sum is within 5e-5 of the oracle's on such islands
    H = plan.amplitude_host(xyz)
    torch.cuda.synchronize()
    assert np.array_equal(A.view(np.float32), H.numpy().reshape(-1).view(np.float32))
    pts = W.grid_points(axes)
    idx = np.random.default_rng(308).choice(len(pts), 150, replace=False)
    ref = oracle.dwba(xyz, pts[idx], c.coef, A_LAT, species=c.species, **gid)
    scale = np.sqrt(np.mean(np.abs(D) ** 2))
    assert np.sqrt(np.mean(np.abs(A[idx] - ref) ** 2)) < 1e-4 * max(scale, np.sqrt(np.mean(np.abs(ref) ** 2)))
    far = xyz.copy()
    far[11, :2] *= 9.0
    assert torch.equal(plan.amplitude(_t(far)), bare.amplitude(_t(far)))
    assert torch.equal(plan.intensity(_t(xyz)), bare.intensity(_t(xyz)))
    plan.check()
