"""The factorised grid sum with tabulated tiles (larger sums) against the oracle, with
odd numbers of columns per thread, without mirror columns, over several species
and with exact phases (past 128 cycles, along the rows and along the columns), and
bit for bit against the tiles that small sums form themselves: a crystal and the same
one with weightless atoms after it, in one chunk.  Tolerance 1e-5, the FP32 sums'."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


def _t(v):
    return torch.tensor(v, device="cuda:0")


def _axes(shape, uneven, steps=None, centre=(0.01, -0.02, 4.0)):
    rng = np.random.default_rng(611)
    steps = steps or [0.9 / n for n in shape]
    axes = [W.linspace_axis(x, n, step=s) for x, n, s in zip(centre, shape, steps)]
    return [a + rng.uniform(-0.2, 0.2, len(a)) * s if u else a for a, s, u in zip(axes, steps, uneven)]


def _plan(coef, n, axes, sp=None, split=0):
    # a hint past which no axis is oversampled: the sum on the map's own points
    return api.Plan(coef, A_LAT, n, axes=axes, atom_species=sp, path="generic", radius_hint=1e6, split_k=split)


@pytest.mark.parametrize("shape, uneven, columns", [
    ((60, 40, 33), (0, 0, 0), None),
    ((200, 9, 60), (1, 0, 1), 10),    # five columns per thread, each with its mirror
    ((120, 13, 61), (1, 0, 1), 14),   # seven
    ((150, 5, 70), (1, 1, 1), 7),     # seven without mirrors
    ((61, 47, 32), (1, 1, 1), None),
])
@pytest.mark.parametrize("crystal", ["sphere", "rod_rows", "rod_columns"])
def test_tabulated_sums(crystal, shape, uneven, columns):
    rng = np.random.default_rng(612)
    if crystal == "sphere":
        c = W.fcc_sphere(radius_cells=15.0, seed=613)
        xyz, sp, coef = c.xyz + np.array([12.3, -4.4, 7.0]), c.species, c.coef
    else:
        # 400 cells: phases past 128 cycles along the long axis of the grid (rows) or along the short one
        long = 0 if crystal == "rod_rows" else 1
        c = W.strained_cube(n=tuple(400 if d == long else 5 for d in range(3)), seed=614)
        xyz, sp, coef = c.xyz, None, c.coef
    occ = rng.uniform(0.5, 1.0, len(xyz)).astype(np.float32)
    axes = _axes(shape, uneven)
    plan = _plan(coef, len(xyz), axes, sp)
    if columns:
        assert plan.info()["points_per_thread"] == columns
    A = plan.amplitude(_t(xyz), _t(occ)).cpu().numpy()
    plan.check()
    S = W.grid_points(axes)
    idx = np.concatenate([rng.choice(len(S), 500, replace=False), np.argsort(np.abs(A))[-20:]])
    ref = oracle.amplitude(xyz, S[idx], coef, A_LAT, species=sp, occ=occ)
    assert np.linalg.norm(A[idx] - ref) < 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("shape, uneven", [((61, 47, 33), (0, 0, 0)), ((200, 9, 60), (1, 0, 1)), ((150, 5, 70), (1, 1, 1)),
                                           ((61, 47, 32), (1, 1, 1))])
@pytest.mark.parametrize("length", [12.0, 400.0])
def test_tables_equal_self_formed_tiles(shape, uneven, length):
    rng = np.random.default_rng(615)
    n, more = 1024, 120 * 1024
    box = np.array([length, 9.0, 9.0])
    xyz = rng.uniform(-0.5, 0.5, (n, 3)) * box
    xyz[0], xyz[1] = 0.5 * box, -0.5 * box
    axes = _axes(shape, uneven)
    coef = W.unit_species()[None]
    small, large = _plan(coef, n, axes, split=1), _plan(coef, more, axes, split=1)
    i, j = small.info(), large.info()
    assert (i["threads"], i["points_per_thread"], i["split_k"]) == (j["threads"], j["points_per_thread"], j["split_k"])
    # records, rounding errors and at least a column's entries per slot beside the position tables
    grown = (j["workspace_bytes"] - i["workspace_bytes"]) / (more - n)
    assert grown > 44 + 24 + 16
    w = rng.uniform(0.5, 1.0, n).astype(np.float32)
    A = small.amplitude(_t(xyz), _t(w))
    both = np.concatenate([xyz, rng.uniform(-0.4, 0.4, (more - n, 3)) * box])
    B = large.amplitude(_t(both), _t(np.concatenate([w, np.zeros(more - n, np.float32)])))
    assert torch.equal(A, B)
