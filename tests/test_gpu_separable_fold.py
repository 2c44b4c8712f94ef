"""The folded separable forward (axes symmetric about their middles) against
the oracle: M tiles of 32 mirror pairs of h values or of 64 h values (one,
several, an odd pair of tiles), column tiles of 128 mirror pairs of points,
odd middles, the in-kernel A tiles, off-centre maps and crystals, and the host
call.  A given split_k keeps the plan on the folded form.
Tolerance: the 1e-4 of the separable map."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A
TOL = 1e-4


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _sphere(seed):
    return W.fcc_sphere(radius_cells=6.6, shell_cells=2.0, seed=seed)  # above the fold's smallest crystal


@pytest.mark.parametrize("split", [1, 3])
@pytest.mark.parametrize("shape, centre, offset", [
    ((1, 1, 1), (0.0, 0.0, 4.0), (0, 0, 0)),
    ((2, 1, 129), (0.0, 0.0, 4.0), (0, 0, 0)),          # one alpha; 65 pairs, one past a column group
    ((5, 3, 85), (0.013, -0.02, 3.97), (0, 0, 0)),      # odd middles; 128 pairs: one full column tile
    ((63, 16, 16), (0.0, 0.0, 4.0), (0, 0, 0)),         # 32 alphas: one full M tile
    ((65, 7, 37), (0.01, 0.0, 4.02), (31, -18, 8)),     # 33 alphas; 130 pairs; off-centre crystal
    ((130, 1, 200), (0.0, 0.0, 4.0), (0, 0, 50)),       # 65 alphas, one column tile: A formed in the kernel
    ((200, 2, 9), (0.004, 0.1, 4.0), (0, 0, 0)),        # the same with 9 pairs
    ((140, 20, 31), (0.0, 0.0, 4.0), (-7, 3, 2)),       # three M tiles: the pair kernel on the A table
    ((300, 5, 60), (0.0, 0.0, 4.0), (0, 0, 0)),         # five M tiles: the one-CTA kernel beside it
    ((33, 9, 30), (0.06, 0.0, 4.0), (0, 0, 0)),         # h off its middle: direct h rows, one M tile
    ((97, 1, 11), (0.2, 0.0, 4.0), (3, 0, -9)),         # two M tiles, the second half full
    ((129, 3, 41), (0.3, 0.0, 4.0), (0, 0, 0)),         # three M tiles, one value in the third; A in the kernel
    ((300, 4, 70), (0.4, 0.0, 4.0), (0, 0, 0)),         # five M tiles
])
def test_folded_map_matches_the_oracle(shape, centre, offset, split):
    c = _sphere(41)
    occ = np.random.default_rng(42).uniform(0.5, 1.0, len(c.xyz)).astype(np.float32)
    axes = [W.linspace_axis(x, n, step=0.003) for x, n in zip(centre, shape)]
    xyz = c.xyz + np.array(offset, dtype=np.float64)
    plan = api.Plan(c.coef, A_LAT, len(xyz), axes=axes, atom_species=c.species, path="separable", split_k=split)
    x, w = torch.tensor(xyz, device="cuda:0"), torch.tensor(occ, device="cuda:0")
    A = plan.amplitude(x, w)
    I = plan.intensity(x, w)
    plan.check()
    S = W.grid_points(axes)
    idx = np.arange(len(S)) if len(S) <= 700 else np.random.default_rng(43).choice(len(S), 700, replace=False)
    ref = oracle.amplitude(xyz, S[idx], c.coef, A_LAT, species=c.species, occ=occ)
    An = A.cpu().numpy()
    assert np.all(np.isfinite(An.view(np.float32)))
    assert _rel(An[idx], ref) < TOL
    assert _rel(I.cpu().numpy()[idx], np.abs(ref) ** 2) < 2 * TOL
    out = plan.amplitude_host(torch.tensor(xyz), torch.tensor(occ))
    torch.cuda.synchronize()
    assert torch.equal(out, A.cpu())


def test_wide_axes_take_the_reduced_and_exact_phases():
    """k spans +-3 r.l.u. (phases of ~20 cycles) on a sphere, and l spans
    +-0.4 over a 600-cell chain of blocks (phases past 128 cycles)."""
    c = _sphere(44)
    axes = [np.linspace(-0.05, 0.05, 5), np.linspace(-3.0, 3.0, 61), np.linspace(3.9, 4.1, 17)]
    plan = api.Plan(c.coef, A_LAT, len(c.xyz), axes=axes, atom_species=c.species, path="separable", split_k=2)
    A = plan.amplitude(torch.tensor(c.xyz, device="cuda:0")).cpu().numpy()
    assert _rel(A, oracle.amplitude(c.xyz, W.grid_points(axes), c.coef, A_LAT, species=c.species)) < TOL
    rod = W.strained_cube(n=(2, 2, 600), seed=45)
    axes = [np.linspace(-0.1, 0.1, 4), np.linspace(-0.1, 0.1, 3), np.linspace(3.6, 4.4, 201)]
    plan = api.Plan(rod.coef, A_LAT, len(rod.xyz), axes=axes, path="separable", split_k=2)
    A = plan.amplitude(torch.tensor(rod.xyz, device="cuda:0")).cpu().numpy()
    assert _rel(A, oracle.amplitude(rod.xyz, W.grid_points(axes), rod.coef, A_LAT)) < TOL


def test_uneven_axis_takes_the_direct_form():
    c = _sphere(46)
    axes = [W.linspace_axis(0.0, 20, step=0.004), np.sort(np.random.default_rng(47).uniform(-0.05, 0.05, 9)),
            W.linspace_axis(4.0, 15, step=0.004)]
    plan = api.Plan(c.coef, A_LAT, len(c.xyz), axes=axes, atom_species=c.species, path="separable")
    A = plan.amplitude(torch.tensor(c.xyz, device="cuda:0")).cpu().numpy()
    assert _rel(A, oracle.amplitude(c.xyz, W.grid_points(axes), c.coef, A_LAT, species=c.species)) < TOL

