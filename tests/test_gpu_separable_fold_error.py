"""Folded tensor-core maps of coherent crystals are no further from the oracle than the
direct form's (which intensities take): relative L2 errors of |A|^2 and of the intensity
over the map, from 20,000 of its points.  Allowed 1.15 times, the scatter of the two
forms' truncations (they round different sums)."""
import numpy as np
import pytest

import oracle
from paper_1010_2641_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_1010_2641_gb300 import api

A_LAT = W.LATTICE_A


@pytest.mark.parametrize("cells, shape, step, off", [
    (14.4, (92, 58, 102), 0.0016, 0.0), (15.6, (56, 92, 85), 0.0026, 0.03), (14.5, (196, 98, 46), 0.0018, 0.05),
    (13.5, (136, 117, 54), 0.0032, -0.04), (12.0, (200, 60, 60), 0.002, 0.05),
])
def test_error_of_the_folded_form(cells, shape, step, off):
    c = W.fcc_sphere(radius_cells=cells, shell_cells=1.0, strain=0.0, seed=621)
    axes = [W.linspace_axis(x + off * n * step, n, step=step) for x, n in zip((0.0, 0.0, 4.0), shape)]
    coef = W.unit_species()[None]
    plan = api.Plan(coef, A_LAT, len(c.xyz), axes=axes, path="separable", radius_hint=1e5)  # without nodes
    x = torch.tensor(c.xyz, device="cuda:0")
    A, I = plan.amplitude(x).cpu().numpy().astype(np.complex128), plan.intensity(x).cpu().numpy().astype(np.float64)
    plan.check()
    J = np.abs(A) ** 2
    assert np.abs(J - I).max() > 1e-6 * I.max()  # folded
    S = W.grid_points(axes)
    idx = np.random.default_rng(622).choice(len(S), 20000, replace=False)
    ref = np.abs(oracle.amplitude(c.xyz, S[idx], coef, A_LAT)) ** 2
    folded, direct = np.linalg.norm(J[idx] - ref), np.linalg.norm(I[idx] - ref)
    assert folded < 1.15 * direct
    assert direct < 2e-4 * np.linalg.norm(ref)
