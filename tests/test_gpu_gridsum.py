"""The factorised FP32 grid sum against the oracle: each axis as the columns,
one to eight columns per thread with and without mirror columns and middles,
rows below and past a block, several species, occupancies, chunks, off-centre
crystals, exact phases, factor tables, no atoms.  Tolerance 1e-5: MUFU
sin/cos (2^-21 absolute per term) and FP32 sums blocked by 128 atoms, ten times
inside the FP32 paths' 1e-4."""
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


@pytest.mark.parametrize("uneven", [False, True])
@pytest.mark.parametrize("shape, split", [
    ((1, 1, 64), 0), ((1, 63, 1), 3), ((129, 1, 1), 0), ((40, 2, 3), 2),         # few rows, the long axis as columns
    ((7, 9, 1), 0), ((7, 9, 2), 0), ((9, 8, 3), 0), ((16, 16, 7), 4),             # few columns
    ((13, 11, 17), 0), ((20, 13, 19), 1), ((33, 8, 20), 5), ((5, 52, 6), 64),     # ragged columns, many chunks
])
def test_grid_matches_the_oracle(shape, split, uneven):
    c = W.fcc_sphere(radius_cells=3.7, seed=81)
    xyz = c.xyz + np.array([12.3, -4.4, 7.0])
    occ = np.random.default_rng(82).uniform(0.5, 1.0, len(xyz)).astype(np.float32)
    axes = [W.linspace_axis(x, n, step=0.013) for x, n in zip((0.01, -0.3, 4.2), shape)]
    if uneven:
        axes = [a + np.random.default_rng(83 + d).uniform(-0.004, 0.004, len(a)) for d, a in enumerate(axes)]
    plan = api.Plan(c.coef, A_LAT, len(xyz), axes=axes, atom_species=c.species, path="generic", split_k=split)
    A, I = plan.amplitude(_t(xyz), _t(occ)), plan.intensity(_t(xyz), _t(occ))
    plan.check()
    ref = oracle.amplitude(xyz, W.grid_points(axes), c.coef, A_LAT, species=c.species, occ=occ)
    assert _rel(A.cpu().numpy(), ref) < TOL
    assert _rel(I.cpu().numpy(), np.abs(ref) ** 2) < 2 * TOL


@pytest.mark.parametrize("cells, axis", [((2, 2, 400), 2), ((400, 2, 2), 0)])
def test_long_crystal_takes_exact_phases(cells, axis):
    """A 400-cell rod along the columns (their table's products are exact) and
    along the rows (phases past 128 cycles: the exact form)."""
    c = W.strained_cube(n=cells, seed=84)
    half = [np.linspace(-0.45, 0.45, 9) if d == axis else np.linspace(-0.1, 0.1, 6) for d in range(3)]
    axes = [half[0], half[1], 4.0 + half[2]]
    plan = api.Plan(c.coef, A_LAT, len(c.xyz), axes=axes, path="generic")
    A = plan.amplitude(_t(c.xyz)).cpu().numpy()
    assert _rel(A, oracle.amplitude(c.xyz, W.grid_points(axes), c.coef, A_LAT)) < TOL


def test_factor_table_and_no_atoms():
    m = W.fcc_cell_blocks(n=(6, 5, 4))
    axes = [np.linspace(-0.06, 0.06, 9), np.linspace(-0.05, 0.05, 7), np.linspace(3.92, 4.08, 12)]
    S = W.grid_points(axes)
    rng = np.random.default_rng(85)
    T = rng.normal(size=(2, len(S))) + 1j * rng.normal(size=(2, len(S)))
    plan = api.Plan(W.si_ge_species(), A_LAT, len(m.origins), axes=axes, atom_species=m.types, path="generic",
                    factor_table=T)
    A = plan.amplitude(_t(m.origins)).cpu().numpy()
    assert _rel(A, oracle.amplitude_table(m.origins, S, T, types=m.types)) < TOL
    empty = api.Plan(W.unit_species()[None], A_LAT, 0, axes=axes, path="generic")
    assert torch.all(empty.amplitude(torch.empty(0, 3, dtype=torch.float64, device="cuda:0")) == 0)
