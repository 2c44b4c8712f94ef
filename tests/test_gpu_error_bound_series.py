"""scatter_error_bound where a plan sums over clusters of points or at Chebyshev
nodes: the error of one term (a crystal with one atom of weight 1, at the radius in
question, the others of weight 0) stays below the bound in every direction, along
the points' principal axes and their diagonals, where clusters and nodes are worst."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


def _directions(S):
    V = np.linalg.svd(S - S.mean(0), full_matrices=False)[2]
    d = [V[0], V[1], V[2], V[0] + V[1], V[0] - V[1], V[0] + V[2], V[1] + V[2], V[0] + V[1] + V[2], V[0] + 0.5 * V[1],
         0.5 * V[0] + V[1]] + list(np.random.default_rng(561).normal(size=(10, 3)))
    return [v / np.linalg.norm(v) for v in d]


def _worst(plan, S, n, radius):
    base = np.random.default_rng(562).uniform(-2.0, 2.0, (n, 3))
    occ = np.zeros(n, np.float32)
    occ[3] = 1.0
    w = torch.tensor(occ, device="cuda:0")
    worst = 0.0
    for u in _directions(S):
        xyz = base.copy()
        xyz[3], xyz[4] = u * radius, -u * radius  # the weightless one keeps the crystal centred
        A = plan.amplitude(torch.tensor(xyz, device="cuda:0"), w).cpu().numpy()
        worst = max(worst, np.abs(A - np.exp(2j * np.pi * (S @ xyz[3]))).max())
    plan.check()
    return worst


@pytest.mark.parametrize("points, half, flat", [(40000, 0.02, 0.3), (10000, 0.04, 0.3), (10000, 0.01, 0.02), (40000, 0.08, 0.3)])
def test_clusters(points, half, flat):
    n = 20000
    S = np.array([1.0, 1.0, 1.0]) + np.random.default_rng(563).uniform(-half, half, (points, 3)) * np.array([1.0, 1.0, flat])
    plan = api.Plan(W.unit_species()[None], A_LAT, n, s_list=S)
    X = 1.45 * np.cbrt(3 * n / (16 * np.pi)) + 1.0
    for part in (0.999, 0.7, 0.4):
        bound, rel = plan.error_bound(part * X)
        err = _worst(plan, S, n, part * X)
        assert err < bound
        assert rel <= bound + 1e-5


@pytest.mark.parametrize("path, shape, step", [("generic", (61, 47, 33), 0.004), ("separable", (129, 130, 65), 0.002),
                                               ("generic", (300, 1, 200), 0.001)])
def test_nodes(path, shape, step):
    n = 45000 if path == "separable" else 20000
    axes = [W.linspace_axis(x, m, step=step) if m > 1 else np.array([x]) for x, m in zip((0.0, 0.0, 4.0), shape)]
    S = W.grid_points(axes)
    plan = api.Plan(W.unit_species()[None], A_LAT, n, axes=axes, path=path)
    bare = api.Plan(W.unit_species()[None], A_LAT, n, axes=axes, path=path, radius_hint=1e5)
    assert plan.info()["workspace_bytes"] > bare.info()["workspace_bytes"]
    compact = np.cbrt(3 * n / (16 * np.pi))
    for radius in (1.1 * compact + 0.99, 1.1 * compact - 3.0):
        bound, rel = plan.error_bound(radius)
        assert _worst(plan, S, n, radius) < bound
        # the interpolation's own error, 1e-6 (FP32 5e-8) per axis and times 10 to 50 along the others
        assert bare.error_bound(radius)[1] < rel < bare.error_bound(radius)[1] + (2e-4 if path == "separable" else 1e-5)


def test_diffuse_map_stays_below_the_model():
    rng = np.random.default_rng(564)
    n = 20000
    u = rng.normal(size=(n, 3))
    xyz = u / np.linalg.norm(u, axis=1, keepdims=True) * 16.0 * np.cbrt(rng.uniform(0.0, 1.0, (n, 1)))
    S = np.array([1.0, 1.0, 1.0]) + rng.uniform(-0.03, 0.03, (30000, 3)) * np.array([1.0, 1.0, 0.3])
    plan = api.Plan(W.unit_species()[None], A_LAT, n, s_list=S)
    sel = rng.choice(len(S), 800, replace=False)
    A = plan.amplitude(torch.tensor(xyz, device="cuda:0")).cpu().numpy()[sel]
    ref = oracle.amplitude(xyz, S[sel], W.unit_species()[None], A_LAT)
    assert np.linalg.norm(A - ref) < plan.error_bound(16.1)[1] * np.linalg.norm(ref)
