"""The tensor-core adjoint over a folded (k, l) plane and its direct form, from
a given amplitude map (the oracle's), against the oracle's analytic gradient:
odd and even planes (with and without a middle point), one k value, planes of
one and of several 16-point steps, middles off H, uneven axes and off-centre
crystals.  Tolerance 1e-4: the contraction's error (f16 hi + lo products,
FP32 accumulation over at most 256 steps), the forward's is not in it."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


@pytest.mark.parametrize("uneven", [False, True])
@pytest.mark.parametrize("shape, centre, offset", [
    ((1, 1, 1), (0.0, 0.0, 4.0), (0, 0, 0)),
    ((3, 1, 32), (0.0, 0.0, 4.0), (0, 0, 0)),           # 16 pairs: one step
    ((5, 3, 11), (0.02, 0.01, 3.99), (0, 0, 0)),        # 17 pairs with a middle point, middles off H
    ((50, 8, 9), (0.0, 0.0, 4.0), (40, -7, 13)),        # several steps; three M tiles of rows; off-centre crystal
    ((70, 5, 9), (0.0, 0.02, 4.02), (0, 0, -9)),        # four M tiles
])
def test_gradient_from_a_given_map(shape, centre, offset, uneven):
    c = W.fcc_sphere(radius_cells=3.1, seed=61)
    xyz = c.xyz + np.array(offset, dtype=np.float64) + 0.2
    occ = np.random.default_rng(62).uniform(0.5, 1.0, len(xyz)).astype(np.float32)
    axes = [W.linspace_axis(x, n, step=0.02) for x, n in zip(centre, shape)]
    if uneven:
        axes[1] = axes[1] + np.random.default_rng(63).uniform(-0.006, 0.006, len(axes[1]))
    S = W.grid_points(axes)
    A = oracle.amplitude(xyz, S, c.coef, A_LAT, species=c.species, occ=occ).astype(np.complex64)
    I_obs = (np.abs(A) ** 2 * np.random.default_rng(64).uniform(0.7, 1.3, len(A))).astype(np.float32)
    plan = api.Plan(c.coef, A_LAT, len(xyz), axes=axes, atom_species=c.species, path="separable")
    t = lambda v: torch.tensor(v, device="cuda:0")
    _, grad = plan.backward(t(xyz), t(A), t(I_obs), t(occ))
    plan.check()
    sel = np.random.default_rng(65).choice(len(xyz), 64, replace=False)
    ref = oracle.loss_grad_atoms(xyz, S, A.astype(np.complex128), I_obs, c.coef, A_LAT, sel, species=c.species, occ=occ)
    ref = ref[1] if isinstance(ref, tuple) else ref
    g = grad.cpu().numpy().astype(np.float64)[sel]
    assert np.linalg.norm(g - ref) < 1e-4 * np.linalg.norm(ref)
